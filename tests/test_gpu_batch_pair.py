"""Two batches alive at once: one whose tiles take little shared memory, made after one whose
tiles take much, must not lower the kernel's limit under the other's launch."""

import numpy as np
import pytest

from oracle import operator as O
from paper_1802_10323_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("order", [(512, 16), (16, 512)])
def test_two_batches(lib, order):
    import torch
    made = []
    for n in order:
        g = dict(nx=n, ny=n // 2, nz=6, dx=1.0 / n, dy=2.0 / n, zf=synth.tanh_faces(6, 1.0, 1.2),
                 bcs=("P", "NN", "DD"), alpha=0.0)
        b = lib.Batch([g], rtol=1e-10, max_iter=6)
        f = torch.as_tensor(np.random.default_rng(n).uniform(-1, 1, (6, n // 2, n)), device="cuda").contiguous()
        p = torch.zeros_like(f)
        made.append((g, b, f, p, b.pointers([f], [p]), lib.infos_tensor(1)))
    for g, b, f, p, (fptr, pptr), infos in made:
        b.solve(fptr, pptr, infos)
    torch.cuda.synchronize()
    for g, b, f, p, _, infos in made:
        assert lib.read_infos(infos, 1)[0].status == 0
        rr = O.relative_residual(p.cpu().numpy(), f.cpu().numpy(), g["dx"], g["dy"], g["zf"], *g["bcs"])
        terms = 4 * (g["dx"] ** -2 + g["dy"] ** -2 + np.diff(g["zf"]).min() ** -2)
        assert rr <= 1e-10 + 2.0 ** -46 * terms * float(p.abs().max() / f.abs().max())
        b.close()
