"""A planar flow (no out-of-plane velocity or field) in a two-dimensional FP64
box, through each kernel that takes one: the kernel of a single box with the plain
Riemann solvers; the batch, learned-switch and characteristic kernels with
the solvers of fewer operations.  The states agree to rounding (1e-13 over ten
steps, the FP64 tolerance between kernels), and the out-of-plane momentum and
field stay rounding: each step adds at most a few eps of products of order
one, 1e-14 over ten steps."""
import numpy as np
import pytest

from helpers import state_errors
from paper_2606_12753_gb300 import inputs as I
from paper_2606_12753_gb300 import mhd, switch_train

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("riemann", ["hlld", "hll"])
def test_planar_flow_in_every_kernel(riemann):
    box, dt, n, got = I.orszag_tang_2d(64), 1e-3, 10, {}

    def run(name, **kw):
        s = mhd.Solver(box, precision="fp64", **kw)
        if kw.get("riemann") == "learned":   # a threshold that every logit, or none, clears
            sw = switch_train.Switch(switch_train.he_init(3))
            s.set_switch(sw.block.data_ptr(), 1e-30 if riemann == "hlld" else 1 - 1e-12)
        s.set_state(box.cell, box.face)
        s.step(dt, n)
        got[name] = s.get_state()
        if kw.get("riemann") == "learned":
            assert s.stats()["faces_hll" if riemann == "hlld" else "faces_hlld"] == 0
        s.close()

    run("single", riemann=riemann)
    run("learned", riemann="learned")
    run("characteristic", riemann=riemann, recon="characteristic")
    b = mhd.Batch([box], "fp64", riemann=riemann)
    b.set_state(0, box.cell, box.face)
    b.step(dt, n)
    got["batch"] = b.get_state(0)
    b.close()
    for name, (c, f) in got.items():
        assert max(np.abs(c[3]).max(), np.abs(f[2]).max()) <= 1e-14, name
        if name != "characteristic":
            assert max(state_errors(c, f, *got["single"]).values()) <= 1e-13, name
