"""The CFL maximum of the FP64 form: a cell forms its speed in FP64 only where
an FP32 estimate says that it may raise the maximum, so the dt of the fused
step and of the standalone reduction must be the largest speed of all cells
as FP64 numpy finds it, also where a fast speed's root cancels (B along one
axis with gamma p = B^2), where one cell holds the maximum, and at scales
beyond FP32's range.  Tolerance: 40 roundings (1e-14); the plain fast speed
loses half its digits where its root cancels, so that state allows 1e-8."""
import numpy as np
import pytest

from paper_2606_12753_gb300 import inputs as I
from paper_2606_12753_gb300 import mhd

pytestmark = pytest.mark.gpu


def _dt(box):
    """cfl / max over cells, FP64 numpy (periodic box)."""
    rho, m, e = box.cell[0], box.cell[1:4], box.cell[4]
    b = [0.5 * (f + np.roll(f, -1, axis=2 - d)) for d, f in enumerate(box.face)]
    p = np.maximum((box.gamma - 1) * (e - 0.5 * (m ** 2).sum(0) / rho - 0.5 * sum(q * q for q in b)), 1e-300)
    a2, b2 = box.gamma * p / rho, sum(q * q for q in b) / rho
    speed = 0
    for d, (n, h) in enumerate(((box.nx, box.dx), (box.ny, box.dy), (box.nz, box.dz))):
        if n > 1:
            x = a2 - b2   # the root without cancellation: (a2 - b2)^2 + 4 a2 (b2 - bn2)
            root = np.sqrt(x * x + 4 * a2 * (b2 - b[d] ** 2 / rho))
            speed = speed + (np.abs(m[d] / rho) + np.sqrt(0.5 * (a2 + b2 + root))) / h
    return box.cfl / speed.max()


@pytest.mark.parametrize("dims", [(16, 8, 4), (37, 21, 40), (70, 33, 1)])
@pytest.mark.parametrize("kind", ["random", "peak", "cancelling", "tiny"])
def test_fp64_cfl_dt(dims, kind):
    box = I.random_state(dims, seed=7)
    tol = 1e-14
    if kind == "peak":       # one cell, late in the march, far above the others
        box.cell[4][-1, -1, -1] *= 50.0
    elif kind == "cancelling":
        tol = 1e-8
        for d in range(3):
            box.face[d][...] = 1.0 if d == 0 else 0.0
        box.cell[4] = 1.0 / box.gamma / (box.gamma - 1) + 0.5 * (box.cell[1:4] ** 2).sum(0) / box.cell[0] + 0.5
    elif kind == "tiny":     # pressures and densities below binary32's normal range
        box.cell *= 1e-42
        for f in box.face:
            f *= 1e-21
    s = mhd.Solver(box, precision="fp64", rho_floor=1e-60, p_floor=1e-60)
    s.set_state(box.cell, box.face)
    assert abs(s.cfl_dt() / _dt(box) - 1) <= tol
    s.step(-1.0, 1)   # the recovery of a state set from outside
    assert abs(s.stats()["last_dt"] / _dt(box) - 1) <= tol
    box.cell, box.face = s.get_state()
    want = _dt(box)
    s.step(-1.0, 1)   # the last stage of the step before
    assert abs(s.stats()["last_dt"] / want - 1) <= tol
