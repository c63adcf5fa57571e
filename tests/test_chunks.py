"""The default z-chunk length is chosen from the box's size; the results may
not depend on it.  A step with the default length and with one chunk per
column or odd lengths gives the same bits, for boxes that get one plane per
chunk up to boxes that keep 32, periodic and outflow, and the batch likewise."""
import numpy as np
import pytest

from paper_2606_12753_gb300 import inputs as I
from paper_2606_12753_gb300 import mhd

pytestmark = pytest.mark.gpu


def _run(box, precision, tz, **kw):
    s = mhd.Solver(box, precision=precision, tile=(0, 0, tz), **kw)
    s.set_state(box.cell, box.face)
    s.step(-1.0, 2)
    c, f = s.get_state()
    s.close()
    return [c] + f


@pytest.mark.parametrize("precision", ["fp64", "mixed", "fp32"])
@pytest.mark.parametrize("dims,bc", [((17, 9, 3), (0, 0, 0)), ((24, 24, 24), (0, 0, 1)), ((64, 40, 50), (0, 0, 0)),
                                     ((33, 70, 2), (1, 1, 1))])
@pytest.mark.parametrize("form", ["rk2", "rk3", "characteristic"])
def test_chunk_length_leaves_the_bits(precision, dims, bc, form):
    kw = {"rk2": {}, "rk3": {"integrator": "rk3"}, "characteristic": {"recon": "characteristic"}}[form]
    box = I.random_state(dims, seed=3, bc=bc)
    ref = _run(box, precision, 0, **kw)
    for tz in (1, 7, dims[2]):
        for a, b in zip(ref, _run(box, precision, tz, **kw)):
            assert np.array_equal(a, b), tz


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_batch_chunk_length_leaves_the_bits(precision):
    boxes = [I.random_state(d, seed=i, bc=(1, 0, 1)) for i, d in enumerate([(20, 17, 30), (9, 33, 5), (40, 8, 61)])]
    got = []
    for tz in (0, 3, 64):
        b = mhd.Batch(boxes, precision, tile=(0, 0, tz))
        for i, q in enumerate(boxes):
            b.set_state(i, q.cell, q.face)
        b.step(-1.0, 2)
        got.append([x for i in range(len(boxes)) for c, f in [b.get_state(i)] for x in [c] + f])
        b.close()
    for other in got[1:]:
        for x, y in zip(got[0], other):
            assert np.array_equal(x, y)
