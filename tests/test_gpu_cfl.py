"""The CFL maximum: a cell forms its speed in FP64 only where an FP32 estimate
says that it may raise the maximum, so the dt of the standalone reduction
(every form) and of the fused FP64 step must be the largest speed of all cells
as FP64 numpy finds it, also where a fast speed's root cancels (B along one
axis with gamma p = B^2), where one cell holds the maximum, where the energy
is almost all magnetic or kinetic, and at scales beyond FP32's range.
Tolerance: 40 roundings (1e-14) times the energy over the thermal energy of
the fastest cell (at most 2e3 here); the fused step's fast speed loses half
its digits where its root cancels, so that state allows it 1e-8."""
import numpy as np
import pytest

from paper_2606_12753_gb300 import inputs as I
from paper_2606_12753_gb300 import mhd

pytestmark = pytest.mark.gpu


def _dt(box):
    """cfl / max over cells, FP64 numpy."""
    cell = box.cell.astype(np.float64)
    rho, m, e = cell[0], cell[1:4], cell[4]
    face = [f.astype(np.float64) for f in box.face]
    face = [f if box.bc[d] else np.concatenate([f, f.take([0], axis=2 - d)], axis=2 - d) for d, f in enumerate(face)]
    b = [0.5 * (f.take(range(f.shape[2 - d] - 1), axis=2 - d) + f.take(range(1, f.shape[2 - d]), axis=2 - d))
         for d, f in enumerate(face)]
    p = np.maximum((box.gamma - 1) * (e - 0.5 * (m ** 2).sum(0) / rho - 0.5 * sum(q * q for q in b)), 1e-300)
    a2, b2 = box.gamma * p / rho, sum(q * q for q in b) / rho
    speed = 0
    for d, (n, h) in enumerate(((box.nx, box.dx), (box.ny, box.dy), (box.nz, box.dz))):
        if n > 1:
            x = a2 - b2   # the root without cancellation: (a2 - b2)^2 + 4 a2 (b2 - bn2)
            root = np.sqrt(x * x + 4 * a2 * (b2 - b[d] ** 2 / rho))
            speed = speed + (np.abs(m[d] / rho) + np.sqrt(0.5 * (a2 + b2 + root))) / h
    return box.cfl / speed.max()


@pytest.mark.parametrize("dims,bc", [((16, 8, 4), (0, 0, 0)), ((37, 21, 40), (1, 0, 1)), ((70, 33, 1), (1, 1, 0)),
                                     ((300, 5, 3), (0, 1, 0))])
@pytest.mark.parametrize("kind", ["random", "peak", "cancelling", "magnetic", "kinetic", "tiny"])
@pytest.mark.parametrize("precision", ["fp64", "mixed", "fp32"])
def test_cfl_dt(dims, bc, kind, precision):
    if kind == "tiny" and precision != "fp64":
        pytest.skip("only FP64 holds such scales")
    box = I.random_state(dims, seed=7, bc=bc)
    tol, fused = 1e-14, 1e-14
    if kind == "peak":       # one cell, late in the march, far above the others
        box.cell[4][-1, -1, -1] *= 50.0
    elif kind == "cancelling":
        fused = 1e-8
        for d in range(3):
            box.face[d][...] = 1.0 if d == 0 else 0.0
        box.cell[4] = 1.0 / box.gamma / (box.gamma - 1) + 0.5 * (box.cell[1:4] ** 2).sum(0) / box.cell[0] + 0.5
    elif kind in ("magnetic", "kinetic"):   # thermal energy a thousandth of the rest
        tol = fused = 2e-11
        if kind == "magnetic":
            box.face[1] += 60.0
            box.cell[4] += 60.0 * 30.0 + 60.0 * 0.5 * (box.face[1].take(range(dims[1]), axis=1) - 60.0)
            box.cell[4] += 30.0 * (np.roll(box.face[1], -1, axis=1).take(range(dims[1]), axis=1) - 60.0)
        else:
            box.cell[4] += 60.0 * box.cell[1] + 0.5 * 60.0 ** 2 * box.cell[0]
            box.cell[1] += 60.0 * box.cell[0]
    elif kind == "tiny":     # pressures and densities below binary32's normal range
        box.cell *= 1e-42
        for f in box.face:
            f *= 1e-21
    s = mhd.Solver(box, precision=precision, rho_floor=1e-60 if kind == "tiny" else 1e-10,
                   p_floor=1e-60 if kind == "tiny" else 1e-10)
    s.set_state(box.cell, box.face)
    box.cell, box.face = s.get_state()   # rounded to the form's state
    assert abs(s.cfl_dt() / _dt(box) - 1) <= tol
    if precision != "fp64":
        return
    s.step(-1.0, 1)   # the recovery of a state set from outside
    assert abs(s.stats()["last_dt"] / _dt(box) - 1) <= fused
    box.cell, box.face = s.get_state()
    want = _dt(box)
    s.step(-1.0, 1)   # the last stage of the step before
    assert abs(s.stats()["last_dt"] / want - 1) <= fused


@pytest.mark.parametrize("what", ["rho", "energy", "face"])
@pytest.mark.parametrize("sign", [1.0, -1.0])
@pytest.mark.parametrize("precision", ["fp64", "mixed", "fp32"])
def test_reductions_leave_out_nan(what, sign, precision):
    """Cells that hold a NaN of either sign, in the row of the maximum and elsewhere, stay out of both
    maxima: the values of the state without them, exactly."""
    box = I.random_state((37, 21, 40), seed=11)
    box.cell[4][-1, -1, -1] *= 50.0      # the fastest cell
    box.face[0][-1, -1, 34] += 3.0       # the largest |div B|, in its row
    s = mhd.Solver(box, precision=precision)
    s.set_state(box.cell, box.face)
    want = s.cfl_dt(), s.divb_max()
    nan = np.copysign(np.nan, sign)
    for at in ((-1, -1, 8), (3, 4, 5), (20, 0, 36)):
        (box.cell[0] if what == "rho" else box.cell[4] if what == "energy" else box.face[1])[at] = nan
    s.set_state(box.cell, box.face)
    assert (s.cfl_dt(), s.divb_max()) == want
