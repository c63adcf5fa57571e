"""The CFL maximum in units far from one.  The cells that need no FP64 speed
are found by an FP32 estimate, whose squares leave binary32's range at speeds
of about 1e10 and of 1e-10: the dt of the fused FP64 step, of a box of a batch
and of the allocation-free step, and that of the standalone reduction of every
form, must still be cfl over the largest FP64 speed.  The fastest cell, 2 %
above most others, lies late in every march and row.  Tolerance: 40 roundings (1e-14) times the
energy over the thermal energy (below 10)."""
import numpy as np
import pytest

from paper_2606_12753_gb300 import inputs as I
from paper_2606_12753_gb300 import mhd

pytestmark = pytest.mark.gpu

#            rho,   speed, B^2 / p
SCALES = {"fast": (1.0, 1e10, 2.0), "fast, weak field": (1.0, 3e9, 1e-2), "slow": (1.0, 1e-12, 2.0),
          "slow and light": (1e-6, 3e-10, 0.5), "heavy": (1e20, 1e5, 2.0), "light": (1e-20, 1e-2, 2.0),
          "one": (1.0, 1.0, 2.0)}


def _box(dims, rho, speed, field, bc=(0, 0, 0)):
    """Uniform but for v_x, which is larger by a few per cent in the second half of each row and most in the last."""
    box = I.random_state(dims, seed=1, bc=bc)
    p = 0.6 * rho * speed ** 2
    b = np.sqrt(field * p / 3.0)
    for f in box.face:
        f[...] = b
    v = np.full(box.cell.shape[1:], 0.05 * speed)
    v[..., dims[0] // 2:] *= 1.2
    v[-1, -1, -1] *= 1.6
    box.cell[0] = rho
    box.cell[1], box.cell[2], box.cell[3] = rho * v, 0.02 * rho * speed, 0.0
    box.cell[4] = p / (box.gamma - 1) + 0.5 * (box.cell[1:4] ** 2).sum(0) / rho + 1.5 * b * b
    return box


def _dt(box):
    """cfl / max over cells, FP64 numpy, without cancellation in the fast speed's root."""
    rho, m, e = box.cell[0], box.cell[1:4], box.cell[4]
    b = I.cell_b(box.face, (box.nx, box.ny, box.nz), box.bc)
    b2 = [x * x / rho for x in b]
    p = (box.gamma - 1) * (e - 0.5 * (m ** 2).sum(0) / rho - 0.5 * sum(x * x for x in b))
    a2, bb = box.gamma * p / rho, sum(b2)
    speed = 0
    for d, (n, h) in enumerate(((box.nx, box.dx), (box.ny, box.dy), (box.nz, box.dz))):
        if n > 1:
            root = np.sqrt((a2 - bb) ** 2 + 4 * a2 * (bb - b2[d]))
            speed = speed + (np.abs(m[d] / rho) + np.sqrt(0.5 * (a2 + bb + root))) / h
    return box.cfl / speed.max()


def _floors(rho, speed):
    return {"rho_floor": 1e-8 * rho, "p_floor": 1e-8 * rho * speed ** 2}


@pytest.mark.parametrize("scale", SCALES)
@pytest.mark.parametrize("dims,form", [((48, 32, 40), "rk2"), ((48, 32, 40), "rk3"), ((48, 32, 40), "characteristic"),
                                       ((64, 40, 1), "rk2")])
def test_fused_step(scale, dims, form):
    box = _box(dims, *SCALES[scale])
    kw = {"rk2": {}, "rk3": {"integrator": "rk3"}, "characteristic": {"recon": "characteristic"}}[form]
    s = mhd.Solver(box, precision="fp64", **kw, **_floors(*SCALES[scale][:2]))
    s.set_state(box.cell, box.face)
    for _ in range(3):   # the recovery of a state set from outside, then the last stages of steps
        box.cell, box.face = s.get_state()
        want = _dt(box)
        s.step(-1.0, 1)
        assert abs(s.stats()["last_dt"] / want - 1) <= 1e-14


@pytest.mark.parametrize("scale", SCALES)
def test_large_box_and_batch(scale):
    """More rows than warps: a later run meets the maximum of the earlier ones."""
    dims = (64, 100, 100)
    box = _box(dims, *SCALES[scale])
    want = _dt(box)
    s = mhd.Solver(box, precision="fp64", **_floors(*SCALES[scale][:2]))
    s.set_state(box.cell, box.face)
    s.step(-1.0, 1)
    assert abs(s.stats()["last_dt"] / want - 1) <= 1e-14
    s.close()
    if min(box.cell[0].min(), box.cell[4].min()) < 1e-6:
        return   # a batch keeps the default floors
    b = mhd.Batch([box, box], "fp64")
    for i in range(2):
        b.set_state(i, box.cell, box.face)
    assert abs(b.box_dt(1) / want - 1) <= 1e-14
    b.step(-1.0, 1)
    box.cell, box.face = b.get_state(1)
    assert abs(b.box_dt(1) / _dt(box) - 1) <= 1e-14
    b.close()


@pytest.mark.parametrize("scale", SCALES)
def test_allocation_free_step(scale):
    import torch
    box = _box((24, 24, 24), *SCALES[scale])
    want = _dt(box)
    cfg = mhd.box_config(box, "fp64")
    cfg.rho_floor, cfg.p_floor = _floors(*SCALES[scale][:2]).values()
    cell = torch.from_numpy(box.cell).cuda()
    face = [torch.from_numpy(f).cuda() for f in box.face]
    oc, of = torch.empty_like(cell), [torch.empty_like(f) for f in face]
    dt = mhd.mhd_step_noalloc(cfg, [c.data_ptr() for c in cell], [f.data_ptr() for f in face],
                              [c.data_ptr() for c in oc], [f.data_ptr() for f in of], -1.0)
    assert abs(dt / want - 1) <= 1e-14


# the standalone reduction, whose FP32 bound subtracts energies: rho, speed, p, pressure floor; the last three hold
# momenta whose squares leave binary32's range, and floors that a pressure lost in infinities would fall to
BOUND = {"fast": (1.0, 1e10, 6e19, 1e10), "slow": (1.0, 1e-12, 6e-25, 1e-33), "heavy": (1e20, 1e5, 6e29, 1e20),
         "dense, fast": (1e14, 1e9, 1e32, 1e10), "dense, slow": (1e25, 1e-3, 1e24, 1e10),
         "supersonic": (1e14, 1e9, 1e28, 1e12)}


@pytest.mark.parametrize("scale", BOUND)
@pytest.mark.parametrize("precision", ["fp64", "mixed", "fp32"])
def test_reduction(scale, precision):
    rho, speed, p, floor = BOUND[scale]
    box = _box((64, 100, 100), rho, speed, 1e-3)
    box.cell[4] += (p - 0.6 * rho * speed ** 2) / (box.gamma - 1)
    s = mhd.Solver(box, precision=precision, p_floor=floor)
    s.set_state(box.cell, box.face)
    cell, face = s.get_state()   # rounded to the form's state
    box.cell, box.face = cell.astype(np.float64), [f.astype(np.float64) for f in face]
    amplified = max(1.0, (box.cell[4] * (box.gamma - 1) / p).max() / 10.0)
    assert abs(s.cfl_dt() / _dt(box) - 1) <= 1e-14 * amplified
