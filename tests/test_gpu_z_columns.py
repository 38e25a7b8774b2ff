"""The z columns at the edges of their kernels.

FP32 columns run in chunks of 16 rows (one kernel for columns of a single chunk, periodic
columns keep their last row aside, so 17 planes are their edge); the low wavenumbers and the
singular column run a warp per column in double-float, on rings of 32 lanes when z is periodic
(n_z ≥ 32); FP64 columns run a warp each on planes of up to 8192 columns and a thread each
beyond. At sizes around those edges, with and without a null space.

The reference takes the oracle's transforms and z coefficients and eliminates the columns in
extended precision with the diagonal formed there: the oracle's own FP64 elimination, whose
b + λ is rounded to FP64, errs by up to ε·‖T_z‖/|λ| (5e-12 at n_z = 65 and λ = −0.07).
Tolerances are those of the solver's other parity tests: FP64 1e-12 of ‖p‖∞, the refined
solve 1e-9 (rtol 1e-10; the constant of a singular problem aside), FP32 5e-5.
"""

import numpy as np
import pytest

from oracle import operator as O
from oracle import solve as S
from paper_1802_10323_gb300 import synth

pytestmark = pytest.mark.gpu

L = np.longdouble


def _thomas(a, b, c, d):
    """a_k x_{k−1} + b_k x_k + c_k x_{k+1} = d_k, columns along the trailing axes, extended precision."""
    cp, x = np.empty_like(d), np.empty_like(d)
    for k in range(len(d)):
        m = b[k] - (a[k] * cp[k - 1] if k else 0)
        cp[k] = c[k] / m
        x[k] = (d[k] - (a[k] * x[k - 1] if k else 0)) / m
    for k in range(len(d) - 2, -1, -1):
        x[k] -= cp[k] * x[k + 1]
    return x


def _reference(f, dx, dy, zf, bcs):
    nz, ny, nx = f.shape
    fh = S.forward_xy(f, bcs[0], bcs[1]).astype(L)
    a, b, c = (v.astype(L) for v in S.z_system(zf, bcs[2]))
    h = np.diff(zf).astype(L)
    if bcs[2] != "FD":  # the diagonal from its terms
        b = -(a + c)
        if bcs[2] in ("DD", "DN"):
            b[0] -= 2 / h[0] ** 2
        if bcs[2] in ("DD", "ND"):
            b[-1] -= 2 / h[-1] ** 2
    B = b[:, None, None] + S.shifts(nx, ny, dx, dy, bcs[0], bcs[1]).astype(L)
    singular = O.is_singular(*bcs)
    if singular:
        B[:, 0, 0] -= 1
    if bcs[2] == "P":  # Sherman–Morrison on the wrap couplings
        ga = -B[0]
        Bp, u = B.copy(), np.zeros_like(fh)
        Bp[0] -= ga
        Bp[-1] -= a[0] * c[-1] / ga
        u[0], u[-1] = ga, c[-1]
        y, z = _thomas(a, Bp, c, fh), _thomas(a, Bp, c, u)
        r = a[0] / ga
        ph = y - (y[0] + r * y[-1]) / (1 + z[0] + r * z[-1]) * z
    else:
        ph = _thomas(a, B, c, fh)
    if singular:  # mean removed, the first unknown pinned, the solution's mean removed
        w = h / h.sum()
        d = fh[:, 0, 0] - (w * fh[:, 0, 0]).sum()
        x = np.zeros(nz, L)
        x[1:] = _thomas(a[1:], b[1:], c[1:], d[1:])
        ph[:, 0, 0] = x - (w * x).sum()
    return S.backward_xy(ph.astype(np.float64), bcs[0], bcs[1])


CASES = [(n, b) for n in (2, 3, 15, 16, 17, 18, 31, 32, 33, 47, 48, 65) for b in ("NN", "P")] + \
        [(16, "DN"), (17, "DD"), (33, "ND"), (64, "DD"), (32, "FD"), (2, "FD")]


@pytest.mark.parametrize("nz,bz", CASES)
@pytest.mark.parametrize("bx,by", [("P", "NN"), ("ND", "P")])
def test_z_columns_match_reference(lib, nz, bz, bx, by):
    import torch
    nx, ny = 32, 24
    bcs = (bx, by, bz)
    zf = synth.uniform_faces(nz, 1.0) if bz == "P" else synth.tanh_faces(nz, 1.0, 1.5)
    dx, dy = 6.0 / nx, 3.0 / ny
    singular = all(b in ("P", "NN") for b in bcs)
    f = synth.uniform_noise((nz, ny, nx), seed=nz, remove_mean=False)
    if bz == "FD":
        f[0] = 0.0
    q = _reference(f, dx, dy, zf, bcs)
    scale = np.abs(q).max()
    for prec, tol, kw in (("fp64", 1e-12, {}), ("fp32", 5e-5, {}),
                          ("fp32_refine", 1e-9, dict(rtol=1e-10, max_iter=6))):
        plan = lib.Plan(nx, ny, nz, dx, dy, zf=zf, bcs=bcs, precision=prec, **kw)
        dt = torch.float32 if prec == "fp32" else torch.float64
        p = plan.solve(torch.as_tensor(f, device="cuda").to(dt).contiguous()).double().cpu().numpy()
        plan.close()
        d = p - q
        if singular and prec == "fp32_refine":
            d = d - d.mean()
        assert np.abs(d).max() <= tol * scale, (prec, np.abs(d).max() / scale)


def test_fp64_columns_beyond_a_warp_each(lib):
    """9216 columns: a thread each, the singular one by a warp of the same launch."""
    import torch
    nx, ny, nz = 96, 96, 40
    zf = synth.tanh_faces(nz, 1.0, 1.5)
    f = synth.uniform_noise((nz, ny, nx), seed=1)
    q = _reference(f, 1.0 / nx, 1.0 / ny, zf, ("NN", "NN", "NN"))
    plan = lib.Plan(nx, ny, nz, 1.0 / nx, 1.0 / ny, zf=zf, bcs=("NN", "NN", "NN"), precision="fp64")
    p = plan.solve(torch.as_tensor(f, device="cuda").contiguous()).cpu().numpy()
    plan.close()
    assert np.abs(p - q).max() <= 1e-12 * np.abs(q).max()
