"""Performance cases: what a user of this solver has it do, through its public entry points.

Every case is one call (or one training/time step) on fields that stay on the GPU: plain
FP64 solves, FP32 solves refined to FP64 accuracy, Helmholtz solves of an implicit
diffusion step, the differentiable projection with its adjoint, RK3 Navier-Stokes steps
and a batch of small grids. Sizes are those of the repository's configurations, tests and
benchmark and of the flows of Table 3 (cavity, channel, duct, Taylor-Green), and generic
ragged ones. Refined pressures whose lowest modes the residual hardly sees (no Dirichlet
end, so that the constant is free, or a periodic z) mostly leave a case in FP32, as the next
program takes them. ``exact`` restates each call in FP64 with plain torch: dense transform
matrices, a Thomas solve and shifted arrays, no code of the package.
"""

import math

import numpy as np
import torch

from paper_1802_10323_gb300 import autograd, binding as lib, synth, workloads

RTOL, MAX_ITER = 1e-10, 4  # the benchmark's refinement target
BATCH_RTOL = 1e-11
DEV = "cuda"


def listed():
    return [
        # The smallest call: one FP64 solve of the 32^3 unit cube. Latency and launches.
        dict(name="fp64 32^3", kind="solve", prec="fp64", nx=32, ny=32, nz=32, bcs="P P NN",
             stretched=False, alpha=0.0, rhs="noise", lx=1.0, ly=1.0),
        # An FP64 solve of the boundary-condition sweep: mixed walls, stretched z.
        dict(name="fp64 256^3", kind="solve", prec="fp64", nx=256, ny=256, nz=256, bcs="DD ND NN",
             stretched=True, alpha=0.0, rhs="smooth", lx=1.0, ly=1.0),
        # A plain FP32 solve on a small ragged box, each axis another pair: a preconditioner
        # or a surrogate model's solve, where FP32 is enough.
        dict(name="fp32 192x96x65", kind="solve", prec="fp32", nx=192, ny=96, nz=65, bcs="DD DN ND",
             stretched=True, alpha=0.0, rhs="noise", lx=1.0, ly=1.0),
        # The headline: the pressure solve of a large channel, refined to 1e-10.
        dict(name="channel 1024^3", kind="solve", prec="fp32_refine", nx=1024, ny=1024, nz=1024, bcs="P P NN",
             stretched=True, alpha=0.0, rhs="div", lx=6.0, ly=3.0),
        # Lines longer than 1024 cells along x and y (a thin layer, open at the top).
        dict(name="long 4096x4096x16", kind="solve", prec="fp32_refine", nx=4096, ny=4096, nz=16, bcs="P P ND",
             stretched=True, alpha=0.0, rhs="noise", lx=6.0, ly=3.0),
        # The triply periodic box of the Taylor-Green vortex, its pressure handed on in FP32.
        dict(name="periodic 512^3", kind="solve", prec="fp32_refine", nx=512, ny=512, nz=512, bcs="P P P",
             stretched=False, alpha=0.0, rhs="div", lx=6.0, ly=6.0, as32=True),
        # A box whose sizes are no powers of two, with a smooth right-hand side (a developed
        # flow's pressure), walls on y and z.
        dict(name="ragged 384x288x201", kind="solve", prec="fp32_refine", nx=384, ny=288, nz=201, bcs="P NN NN",
             stretched=True, alpha=0.0, rhs="smooth", lx=4.0, ly=2.0),
        # Implicit diffusion of a velocity component on the channel grid of Table 3.
        dict(name="helmholtz 512x256x144", kind="solve", prec="fp32_refine", nx=512, ny=256, nz=144, bcs="P P DD",
             stretched=True, alpha=2.0e4, rhs="noise", lx=6.0, ly=3.0),
        # A training step through the projection: forward and vector-Jacobian product, FP32.
        dict(name="projection 512x256x256", kind="projection", prec="fp32", nx=512, ny=256, nz=256, bcs="P P NN",
             stretched=True, lx=6.0, ly=3.0),
        # One RK3 time step (three substeps) of a channel with FP64 fields.
        dict(name="rk3 channel 512x256x256", kind="rk3", prec="fp32_refine", nx=512, ny=256, nz=256, bcs="P P NN",
             stretched=True, lx=6.0, ly=3.0, nu=1.0 / 5600.0),
        # One RK3 time step of the 128^3 cavity: walls on every axis, small launches.
        dict(name="rk3 cavity 128^3", kind="rk3", prec="fp32_refine", nx=128, ny=128, nz=128, bcs="NN NN NN",
             stretched=True, lx=1.0, ly=1.0, nu=1.0 / 1000.0),
        # 64 independent grids of uneven sizes in one persistent launch, tiles autotuned; a grid
        # without a Dirichlet end carries a Helmholtz shift (an implicit diffusion step).
        dict(name="batch 64 grids", kind="batch", count=64, grids_seed=4),
    ]


def _sizes(lo, hi):
    """Line lengths 2 * 2^a * 3^b in [lo, hi]."""
    return sorted(2 * 2 ** a * 3 ** b for a in range(13) for b in range(8) if lo <= 2 * 2 ** a * 3 ** b <= hi)


def _pick(rng, lo, hi):
    t = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return min(_sizes(lo, hi), key=lambda n: abs(math.log(n / t)))


def _box(rng, lo, hi, zlo, zhi, points):
    while True:
        nx, ny = _pick(rng, lo, hi), _pick(rng, lo, hi)
        nz = int(round(math.exp(rng.uniform(math.log(zlo), math.log(zhi)))))
        if nx * ny * nz <= points:
            return dict(nx=nx, ny=ny, nz=nz)


def draw(rng):
    kind = rng.choice(("fp64", "fp32", "refine", "refine", "refine", "helmholtz", "projection", "rk3", "batch"))
    walls, flow = ("NN", "DD", "ND", "DN"), ("P", "NN")
    box = dict(lx=rng.choice((1.0, 2.0, 6.0)), ly=rng.choice((1.0, 3.0)))
    if kind == "batch":
        return dict(kind="batch", count=rng.choice((6, 12, 24, 48, 64)), grids_seed=rng.randrange(1000))
    if kind == "projection":
        return dict(kind="projection", prec="fp32", bcs=" ".join((rng.choice(flow), rng.choice(flow), "NN")),
                    stretched=True, **box, **_box(rng, 48, 1024, 24, 384, 1 << 25))
    if kind == "rk3":
        bcs = [rng.choice(flow), rng.choice(flow), "NN"]
        return dict(kind="rk3", prec="fp32_refine", bcs=" ".join(bcs), stretched=True,
                    nu=rng.choice((1 / 1000.0, 1 / 5600.0)), **box, **_box(rng, 48, 512, 32, 384, 1 << 24))
    if kind == "fp64":
        bcs = [rng.choice(("P",) + walls) for _ in range(3)]
        return dict(kind="solve", prec="fp64", bcs=" ".join(bcs), stretched=bcs[2] != "P", alpha=0.0,
                    rhs=rng.choice(("noise", "smooth")), **box, **_box(rng, 32, 512, 24, 512, 1 << 24))
    if kind == "fp32":
        bcs = [rng.choice(("P",) + walls) for _ in range(2)] + [rng.choice(walls)]
        return dict(kind="solve", prec="fp32", bcs=" ".join(bcs), stretched=True, alpha=0.0, rhs="noise",
                    **box, **_box(rng, 32, 1024, 24, 512, 1 << 25))
    if kind == "helmholtz":
        bcs = [rng.choice(("P",) + walls) for _ in range(3)]
        return dict(kind="solve", prec="fp32_refine", bcs=" ".join(bcs), stretched=bcs[2] != "P",
                    alpha=10.0 ** rng.uniform(2, 6), as32=bcs[2] == "P", rhs="noise", **box, **_box(rng, 64, 1024, 24, 512, 1 << 26))
    bcs = [rng.choice(("P",) + walls) for _ in range(3)]
    div = all(b in flow for b in bcs)
    return dict(kind="solve", prec="fp32_refine", bcs=" ".join(bcs), stretched=bcs[2] != "P", alpha=0.0,
                as32=div or bcs[2] == "P", rhs=rng.choice(("div", "smooth")) if div else rng.choice(("noise", "smooth")), **box,
                **_box(rng, 64, 4096, 16, 768, 1 << 26))


# ---- inputs -----------------------------------------------------------------------------


def _grid(c):
    zf = synth.tanh_faces(c["nz"], 1.0, 1.5) if c["stretched"] else synth.uniform_faces(c["nz"], 1.0)
    return c["lx"] / c["nx"], c["ly"] / c["ny"], zf, tuple(c["bcs"].split())


def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(seed)


def _singular(c, bcs):
    return all(b in ("P", "NN") for b in bcs) and not c.get("alpha")


def _profile(n, bc):
    x = (torch.arange(n, dtype=torch.float64, device=DEV) + 0.5) / n
    arg = {"P": 2 * x, "NN": x, "DD": x, "ND": 0.5 * x, "DN": 0.5 * x}[bc] * math.pi
    return torch.cos(arg) if bc in ("P", "NN", "ND") else torch.sin(arg)


def _rhs(c, seed):
    """A right-hand side [nz, ny, nx], FP64: the discrete divergence of a Gaussian staggered
    velocity ("div", walls carry no normal velocity), U[-1, 1] noise ("noise"), or a smooth
    product of the axes' lowest modes with 10 % noise ("smooth")."""
    dx, dy, zf, bcs = _grid(c)
    shape, g = (c["nz"], c["ny"], c["nx"]), _gen(seed)
    if c["rhs"] == "div":
        u = torch.randn(shape, generator=g, device=DEV, dtype=torch.float64)
        f = _div1(u, 2, bcs[0], dx)
        del u
        f += _div1(torch.randn(shape, generator=g, device=DEV, dtype=torch.float64), 1, bcs[1], dy)
        f += _div1(torch.randn(shape, generator=g, device=DEV, dtype=torch.float64), 0, bcs[2], _col(np.diff(zf)))
        return f
    f = torch.rand(shape, generator=g, device=DEV, dtype=torch.float64).mul_(2.0).sub_(1.0)
    if c["rhs"] == "smooth":
        px, py, pz = (_profile(n, b) for n, b in zip((c["nx"], c["ny"], c["nz"]), bcs))
        f = f.mul_(0.1) + pz[:, None, None] * py[None, :, None] * px[None, None, :]
    return f - f.mean() if _singular(c, bcs) else f


def _velocity(c, seed):
    """Stacked staggered velocity: a laminar channel profile along x where z has walls and x
    none, with Gaussian fluctuations; no normal velocity on the walls."""
    bcs = c["bcs"].split()
    u = torch.randn((3, c["nz"], c["ny"], c["nx"]), generator=_gen(seed), device=DEV, dtype=torch.float64).mul_(0.1)
    if bcs[2] == "NN" and bcs[0] == "P":
        zf = _grid(c)[2]
        zc = torch.as_tensor(0.5 * (zf[1:] + zf[:-1]), device=DEV)
        u[0] += (6.0 * zc * (1.0 - zc))[:, None, None]
    for comp, axis in ((0, 2), (1, 1), (2, 0)):
        if bcs[comp] != "P":
            u[comp].select(axis, 0).zero_()
    return u


def _dt(c):
    """A time step within the advective and viscous limits of the explicit scheme."""
    dx, dy, zf, _ = _grid(c)
    dz = float(np.diff(zf).min())
    return 0.5 / (2.0 / dx + 0.5 / dy + 0.5 / dz + 4.0 * c["nu"] * (dx ** -2 + dy ** -2 + dz ** -2))


def _batch_grids(c):
    grids = workloads.batch_grids(c["count"], seed=c["grids_seed"])
    for d in grids:
        d["alpha"] = 50.0 if all(b in ("P", "NN") for b in d["bcs"]) else 0.0
    return grids


def _batch_rhs(grids, seed):
    g, out = _gen(seed), []
    for d in grids:
        f = torch.rand((d["nz"], d["ny"], d["nx"]), generator=g, device=DEV, dtype=torch.float64)
        out.append(f.mul_(2.0).sub_(1.0))
    return out


def prepare(case, seed):
    c = case
    if c["kind"] == "batch":
        grids = _batch_grids(c)
        batch = lib.Batch(grids, rtol=BATCH_RTOL, max_iter=MAX_ITER)
        f = _batch_rhs(grids, seed)
        p = [torch.zeros_like(x) for x in f]
        fptr, pptr = batch.pointers(f, p)
        infos = lib.infos_tensor(len(grids), DEV)
        batch.autotune(fptr, pptr)
        return dict(kind="batch", batch=batch, f=f, p=p, fptr=fptr, pptr=pptr, infos=infos)
    dx, dy, zf, bcs = _grid(c)
    n = (c["nx"], c["ny"], c["nz"])
    if c["kind"] == "projection":
        proj = autograd.Projection(*n, dx, dy, zf=zf, bcs=bcs, precision=c["prec"])
        u = _velocity(c, seed).float().requires_grad_(True)
        w = torch.randn(u.shape, generator=_gen(seed + 1), device=DEV, dtype=torch.float32)
        proj.plan.workspace(DEV)
        return dict(kind="projection", proj=proj, u=u, w=w)
    plan = lib.Plan(*n, dx, dy, zf=zf, bcs=bcs, precision=c["prec"], rtol=RTOL, max_iter=MAX_ITER,
                    alpha=c.get("alpha", 0.0))
    plan.workspace(DEV)
    info = lib.info_tensor(DEV)
    if c["kind"] == "rk3":
        u = _velocity(c, seed)
        p = torch.zeros(u.shape[1:], dtype=torch.float64, device=DEV)
        return dict(kind="rk3", plan=plan, info=info, dt=_dt(c), nu=c["nu"], u=u, ustar=torch.empty_like(u),
                    ad=torch.zeros_like(u), p=p, phi=torch.empty_like(p), rhs=torch.empty_like(p))
    f = _rhs(c, seed)
    if c["prec"] == "fp32":
        f = f.float()
    return dict(kind="solve", plan=plan, info=info, f=f, out=torch.empty_like(f), as32=c.get("as32", False))


def run(state):
    s = state
    if s["kind"] == "solve":
        p = s["plan"].solve(s["f"], out=s["out"], info=s["info"])
        return p.float() if s["as32"] else p
    if s["kind"] == "batch":
        s["batch"].solve(s["fptr"], s["pptr"], s["infos"])
        return s["p"]
    if s["kind"] == "projection":
        v = s["proj"](s["u"])
        (g,) = torch.autograd.grad(v, s["u"], s["w"])
        return dict(u=v.detach(), grad=g)
    for k in (1, 2, 3):
        s["plan"].ns_substep(k, s["dt"], s["nu"], s["u"], s["ustar"], s["ad"], s["p"], s["phi"], s["rhs"],
                             info=s["info"])
    # (the pressure leaves in FP32, as a snapshot does: its constant is free)
    return dict(u=s["u"], p=s["p"].float())


def work(case):
    """Inputs once, outputs once; flops: four line transforms (a real FFT of n values and its
    pre- and post-processing) and the elimination along z, once per solve."""
    c = case
    if c["kind"] == "batch":
        pts = [(d["nx"], d["ny"], d["nz"]) for d in _batch_grids(c)]
        return dict(bytes=16.0 * sum(x * y * z for x, y, z in pts), flops=sum(_flops(*p) for p in pts))
    n = c["nx"] * c["ny"] * c["nz"]
    one = _flops(c["nx"], c["ny"], c["nz"])
    if c["kind"] == "projection":  # u*, u, the upstream gradient and the gradient, FP32
        return dict(bytes=48.0 * n, flops=2 * (one + 24.0 * n))
    if c["kind"] == "rk3":  # u and p in and out; about 110 flops of each substep's predictor
        return dict(bytes=64.0 * n, flops=3 * (one + 140.0 * n))
    return dict(bytes=(8.0 if c["prec"] == "fp32" else 16.0) * n, flops=one)


def _flops(nx, ny, nz):
    return nx * ny * nz * (5.0 * (math.log2(nx) + math.log2(ny)) + 16.0 + 9.0)


# ---- the same results in FP64, plain torch ------------------------------------------------


def _col(v):
    return torch.as_tensor(np.asarray(v, dtype=np.float64), device=DEV)[:, None, None]


def _basis(n, bc, h):
    """Orthonormal eigenvectors [n, n] (a column per mode) and eigenvalues of the second
    difference of the axis; every angle reduced as an integer multiple of 2*pi/(8n)."""
    j, q = np.arange(n)[:, None], np.arange(n)[None, :]
    if bc == "P":
        l = (q + 1) // 2
        t, odd, th = 8 * l * j, (q % 2 == 0) & (q > 0), 4 * l
    elif bc == "NN":
        t, odd, th = 2 * q * (2 * j + 1), np.zeros_like(q, bool), 2 * q
    elif bc == "DD":
        t, odd, th = 2 * (q + 1) * (2 * j + 1), np.ones_like(q, bool), 2 * (q + 1)
    else:
        t, odd, th = (2 * q + 1) * (2 * j + 1), np.full(q.shape, bc == "DN"), 2 * q + 1
    ang = 2.0 * np.pi / (8 * n)
    t = t % (8 * n) * ang
    v = np.where(odd, np.sin(t), np.cos(t))
    v /= np.sqrt((v * v).sum(axis=0))
    lam = -4.0 * np.sin(th[0] * (np.pi / (4 * n))) ** 2 / h ** 2
    return torch.as_tensor(v, device=DEV), torch.as_tensor(lam, device=DEV)


def _solve64(f, dx, dy, zf, bcs, alpha=0.0):
    nz, ny, nx = f.shape
    vx, lx = _basis(nx, bcs[0], dx)
    vy, ly = _basis(ny, bcs[1], dy)
    w = torch.matmul(vy.T, torch.matmul(f, vx))
    lam = lx[None, :] + ly[:, None] - alpha
    singular = all(b in ("P", "NN") for b in bcs) and alpha == 0.0
    h = np.diff(zf)
    if bcs[2] == "P":  # uniform z: a third transform
        vz, lz = _basis(nz, "P", float(h[0]))
        w = torch.matmul(vz.T, w.reshape(nz, -1)).reshape(nz, ny, nx)
        d = lz[:, None, None] + lam
        if singular:
            d[0, 0, 0] = math.inf
        w = torch.matmul(vz, (w / d).reshape(nz, -1)).reshape(nz, ny, nx)
    else:
        hc = 0.5 * (h[1:] + h[:-1])
        a, c = np.zeros(nz), np.zeros(nz)
        a[1:], c[:-1] = 1.0 / (h[1:] * hc), 1.0 / (h[:-1] * hc)
        b = -(a + c)
        if bcs[2] in ("DD", "DN"):
            b[0] -= 2.0 / h[0] ** 2
        if bcs[2] in ("DD", "ND"):
            b[-1] -= 2.0 / h[-1] ** 2
        hw = torch.as_tensor(h / h.sum(), device=DEV)
        pin = torch.zeros_like(lam)
        if singular:  # the mean removed, the first unknown pinned to 0, its mean removed
            w[:, 0, 0] -= (hw * w[:, 0, 0]).sum()
            w[0, 0, 0] = 0.0
            pin[0, 0] = 1.0
        cp = torch.empty_like(w)
        for k in range(nz):
            m = b[k] + lam
            if k:
                m = m - a[k] * cp[k - 1]
                w[k] -= a[k] * w[k - 1]
            cp[k] = c[k] / m
            w[k] /= m
            if singular and k == 0:
                cp[0, 0, 0] = 0.0
                w[0, 0, 0] = 0.0
        for k in range(nz - 2, -1, -1):
            w[k] -= cp[k] * w[k + 1]
        del cp
        if singular:
            w[:, 0, 0] -= (hw * w[:, 0, 0]).sum()
    return torch.matmul(torch.matmul(vy, w), vx.T)


def _dn(a, ax, bc, normal=False):
    """Neighbour below along an axis: wrapped, 0 below a wall face (normal component), or the
    ghost cell mirrored across a no-slip wall."""
    if bc == "P":
        return torch.roll(a, 1, ax)
    e = a.narrow(ax, 0, 1)
    return torch.cat([torch.zeros_like(e) if normal else -e, a.narrow(ax, 0, a.shape[ax] - 1)], ax)


def _up(a, ax, bc, normal=False):
    if bc == "P":
        return torch.roll(a, -1, ax)
    e = a.narrow(ax, a.shape[ax] - 1, 1)
    return torch.cat([a.narrow(ax, 1, a.shape[ax] - 1), torch.zeros_like(e) if normal else -e], ax)


def _face(a, ax, bc):
    """A face quantity with its wall face 0 set to 0."""
    if bc != "P":
        a = a.clone()
        a.narrow(ax, 0, 1).zero_()
    return a


def _div1(u, ax, bc, h):
    u = _face(u, ax, bc)
    return (_up(u, ax, bc, True) - u) / h


def _metrics(c):
    """Per axis (array axis, boundary pair, width, centre distance below, above)."""
    dx, dy, zf, bcs = _grid(c)
    h = np.diff(zf)
    hc = 0.5 * (h[1:] + h[:-1])
    per = bcs[2] == "P"
    end = 0.5 * (h[0] + h[-1])
    dn = np.concatenate([[end if per else h[0]], hc])
    up = np.concatenate([hc, [end if per else h[-1]]])
    return [(2, bcs[0], dx, dx, dx), (1, bcs[1], dy, dy, dy), (0, bcs[2], _col(h), _col(dn), _col(up))]


def _project64(c, u):
    """(u - G phi, phi) with A phi = D u."""
    dx, dy, zf, bcs = _grid(c)
    m = _metrics(c)
    f = sum(_div1(u[k], ax, bc, h) for k, (ax, bc, h, _, _) in enumerate(m))
    phi = _solve64(f, dx, dy, zf, bcs)
    return torch.stack([u[k] - _face((phi - torch.roll(phi, 1, ax)) / dn, ax, bc)
                        for k, (ax, bc, _, dn, _) in enumerate(m)]), phi


def _advdiff64(c, u3):
    m = _metrics(c)
    u = [_face(u3[k], m[k][0], m[k][1]) for k in range(3)]
    out = []
    for k, (ax, bc, h, dn, _) in enumerate(m):
        v = u[k]
        cc = (0.5 * (v + _up(v, ax, bc, True))) ** 2
        hm = torch.roll(h, 1, 0) if torch.is_tensor(h) else h
        ad = -(cc - torch.roll(cc, 1, ax)) / dn
        ad += c["nu"] * ((_up(v, ax, bc, True) - v) / h - (v - _dn(v, ax, bc, True)) / hm) / dn
        for d, (bx, bd, hd, ddn, dup) in enumerate(m):
            if d != k:
                e = 0.25 * (v + _dn(v, bx, bd)) * (u[d] + _dn(u[d], ax, bc))
                ad -= (_up(e, bx, bd, True) - e) / hd
                ad += c["nu"] * ((_up(v, bx, bd) - v) / dup - (v - _dn(v, bx, bd)) / ddn) / hd
        out.append(_face(ad, ax, bc))
    return out


def exact(case, seed):
    c = case
    if c["kind"] == "batch":
        grids = _batch_grids(c)
        return [_solve64(f, d["dx"], d["dy"], d["zf"], d["bcs"], d["alpha"]) for d, f in zip(grids, _batch_rhs(grids, seed))]
    dx, dy, zf, bcs = _grid(c)
    if c["kind"] == "solve":
        f = _rhs(c, seed)
        return _solve64(f.float().double() if c["prec"] == "fp32" else f, dx, dy, zf, bcs, c["alpha"])
    if c["kind"] == "projection":
        # The projection is self-adjoint under the weights of the face volumes, so its
        # transpose is W P W^-1 (the common factor dx*dy left out).
        u = _velocity(c, seed).float().double()
        w = torch.randn(u.shape, generator=_gen(seed + 1), device=DEV, dtype=torch.float32).double()
        h, dn = _metrics(c)[2][2:4]
        vol = [h, h, dn]
        g = _project64(c, torch.stack([w[k] / vol[k] for k in range(3)]))[0]
        return dict(u=_project64(c, u)[0], grad=torch.stack([g[k] * vol[k] for k in range(3)]))
    u, dt = _velocity(c, seed), _dt(c)
    p, prev, m = torch.zeros_like(u[0]), None, _metrics(c)
    for al, be in ((8 / 15, 0.0), (5 / 12, -17 / 60), (3 / 4, -5 / 12)):
        ga, ad, us = al + be, _advdiff64(c, u), []
        for k, (ax, bc, _, dn, _) in enumerate(m):
            inc = al * ad[k] - ga * _face((p - torch.roll(p, 1, ax)) / dn, ax, bc)
            us.append(u[k] + dt * (inc if prev is None else inc + be * prev[k]))
        u, phi = _project64(c, torch.stack(us))
        p, prev = p + phi / (ga * dt), ad
    return dict(u=u, p=p)
