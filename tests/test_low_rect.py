"""The rectangle of low-wavenumber columns that FP32 plans solve in double-float (csrc/low_rect.h).

Compiled here by the host compiler and compared with all rectangles of a plane, on the oracle's
eigenvalues: none of at most the same size leaves a smaller κ = ‖T_z‖/|λ| outside, it is cut
off where the rule says (κ of 10^3 with few columns, 10^5 beyond, an eighth of the plane), and
no smaller one would have done.
"""

import os
import shutil
import subprocess

import numpy as np
import pytest

from oracle import solve as S
from oracle import transforms as T
from paper_1802_10323_gb300 import synth

HEADER = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1802_10323_gb300", "csrc",
                      "low_rect.h")
FEW = 304
MAIN = r'''
#include "%s"
#include <stdio.h>
int main() {
  int nx, ny, few;
  double alpha, tz;
  while (scanf("%%d %%d %%lf %%lf %%d", &nx, &ny, &alpha, &tz, &few) == 5) {
    std::vector<double> lx(nx), ly(ny);
    for (double& v : lx) if (scanf("%%lf", &v) != 1) return 1;
    for (double& v : ly) if (scanf("%%lf", &v) != 1) return 1;
    int qx = -1, qy = -1;
    ps::low_rectangle(lx, ly, alpha, tz, few, &qx, &qy);
    printf("%%d %%d\n", qx, qy);
  }
  return 0;
}
'''


@pytest.fixture(scope="module")
def rectangles(tmp_path_factory):
    cxx = shutil.which("g++") or pytest.skip("no host compiler")
    d = tmp_path_factory.mktemp("rect")
    (d / "main.cc").write_text(MAIN % HEADER)
    subprocess.run([cxx, "-std=c++17", "-O1", "-o", str(d / "main"), str(d / "main.cc")], check=True)

    def run(cases):
        text = []
        for lx, ly, alpha, tz in cases:
            text.append(f"{len(lx)} {len(ly)} {float(alpha)!r} {float(tz)!r} {FEW}")
            text.append(" ".join(repr(float(v)) for v in lx))
            text.append(" ".join(repr(float(v)) for v in ly))
        out = subprocess.run([str(d / "main")], input="\n".join(text), capture_output=True, text=True, check=True).stdout
        return [tuple(map(int, line.split())) for line in out.splitlines()]
    return run


def _case(nx, ny, nz, bcs, lx, ly, alpha=0.0):
    zf = synth.uniform_faces(nz, 1.0) if bcs[2] == "P" else synth.tanh_faces(nz, 1.0, 1.5)
    a, b, c = S.z_system(zf, bcs[2])
    tz = (np.abs(a) + np.abs(b) + np.abs(c)).max()
    return (T.eigenvalues(bcs[0], nx) / (lx / nx) ** 2, T.eigenvalues(bcs[1], ny) / (ly / ny) ** 2, alpha, tz)


def _outside(case):
    """κ[qx, qy]: the largest of the columns outside the rectangle q_x < qx, q_y < qy."""
    lx, ly, alpha, tz = case
    with np.errstate(divide="ignore"):
        k = tz / (np.abs(lx)[:, None] + np.abs(ly)[None, :] + alpha)
    x = np.append(np.maximum.accumulate(k.max(axis=1)[::-1])[::-1], 0.0)
    y = np.append(np.maximum.accumulate(k.max(axis=0)[::-1])[::-1], 0.0)
    return np.maximum(x[:, None], y[None, :])


def _check(case, qx, qy):
    out = _outside(case)
    nx, ny = len(case[0]), len(case[1])
    area = np.arange(nx + 1)[:, None] * np.arange(ny + 1)[None, :]
    most, k, tol = nx * ny // 8, out[qx, qy], 1 + 1e-12
    assert qx * qy <= most and (qx == 0) == (qy == 0)
    assert k <= out[area <= qx * qy].min() * tol
    if qx * qy <= FEW:
        assert k <= 1e3 * tol or k <= out[area <= min(FEW, most)].min() * tol
    if qx * qy > FEW or k > 1e5:  # grown for 10^5: as far as it goes, and no further than needed
        assert k <= 1e5 * tol or k <= out[area <= most].min() * tol
        assert not (out[area < qx * qy] <= min(k, 1e5) / tol).any()


def test_rectangles_leave_the_smallest_condition_outside(rectangles):
    rng = np.random.default_rng(5)
    sizes, bc = (2, 4, 6, 8, 12, 16, 24, 32, 48, 64, 96, 162), ("P", "NN", "DD", "ND", "DN", "FD")
    cases = []
    for _ in range(400):
        bcs = tuple(str(b) for b in rng.choice(bc, 2)) + (str(rng.choice(bc[:5])),)
        cases.append(_case(int(rng.choice(sizes)), int(rng.choice(sizes)), int(rng.integers(2, 1200)), bcs,
                           float(rng.choice([0.1, 1.0, 2.0, 6.0])), float(rng.choice([1.0, 3.0])),
                           float(rng.choice([0.0, 0.0, 10.0, 1e4]))))
    for case, (qx, qy) in zip(cases, rectangles(cases)):
        _check(case, qx, qy)


# grid, and the largest κ that the rectangle may leave outside
NAMED = [((48, 48, 512, ("NN", "NN", "NN"), 6.0, 3.0), 1.0e5),
         ((32, 32, 512, ("NN", "NN", "NN"), 1.0, 1.0), 1.5e4),
         ((512, 256, 256, ("P", "P", "NN"), 6.0, 3.0), 2.5e4),
         ((1024, 1024, 1024, ("P", "P", "NN"), 6.0, 3.0), 1.0e5),
         ((4096, 4096, 16, ("P", "P", "ND"), 6.0, 3.0), 1.0e3)]


def test_named_grids(rectangles):
    cases = [_case(*g) for g, _ in NAMED]
    for case, (qx, qy), (g, most) in zip(cases, rectangles(cases), NAMED):
        k = _outside(case)[qx, qy]
        print(g, qx, qy, "%.3g" % k)
        assert k <= most, (g, qx, qy, k)


def test_no_rectangle_without_finite_couplings(rectangles):
    lx = T.eigenvalues("NN", 8)
    assert rectangles([(lx, lx, 0.0, tz) for tz in (np.inf, np.nan, 0.0)]) == [(0, 0)] * 3
