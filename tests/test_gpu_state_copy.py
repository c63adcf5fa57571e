"""State copies between the caller's device arrays and a handle run as one
kernel that picks its access width from both ends' alignment: arrays at
every element offset from a 16-byte boundary, of odd and even lengths, shorter
than one access up to several per thread, come back unchanged, through a box
and through a batch (whose primitives of several boxes share a launch)."""
import numpy as np
import pytest

from paper_2606_12753_gb300 import inputs as I
from paper_2606_12753_gb300 import mhd

pytestmark = pytest.mark.gpu


def _device_arrays(arrays, offset):
    """Copies of the arrays in one device buffer, each `offset` elements past a 16-byte boundary."""
    import torch
    per = 16 // arrays[0].itemsize
    out, at = [], 0
    buf = torch.zeros(sum(a.size + 2 * per for a in arrays), dtype=torch.from_numpy(arrays[0]).dtype, device="cuda")
    for a in arrays:
        start = -(-at // per) * per + offset
        out.append(buf[start:start + a.size])
        out[-1].copy_(torch.from_numpy(np.ascontiguousarray(a).ravel()))
        at = start + a.size
    return out


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("dims,bc", [((3, 2, 2), (1, 1, 1)), ((7, 5, 3), (0, 1, 0)), ((64, 48, 33), (1, 0, 0))])
@pytest.mark.parametrize("offset", [0, 1, 2, 3])
def test_device_state_round_trip(precision, dims, bc, offset):
    import torch
    dt = np.float32 if precision == "fp32" else np.float64
    if offset >= 16 // dt(0).itemsize:
        pytest.skip("the same alignment as a smaller offset")
    box = I.random_state(dims, seed=offset, bc=bc)
    arrays = [box.cell[v].astype(dt) for v in range(5)] + [f.astype(dt) for f in box.face]
    src = _device_arrays(arrays, offset)
    dst = [torch.full_like(x, -1.0) for x in _device_arrays(arrays, (offset + 1) % 4)]
    sp, dp = [x.data_ptr() for x in src], [x.data_ptr() for x in dst]
    s = mhd.Solver(box, precision=precision)
    mhd.mhd_set_state(s.h, sp[:5], sp[5:], 1)
    mhd.mhd_get_state(s.h, dp[:5], dp[5:], 1)
    for a, d in zip(arrays, dst):
        assert np.array_equal(a.ravel(), d.cpu().numpy())
    b, lib = mhd.Batch([box, box], precision), mhd.load()
    for x in dst:
        x.fill_(-1.0)
    for i in range(2):
        assert lib.mhd_batch_set_state(b.h, i, (mhd._VP * 5)(*sp[:5]), (mhd._VP * 3)(*sp[5:]), 1) == 0
    assert lib.mhd_batch_get_state(b.h, 1, (mhd._VP * 5)(*dp[:5]), (mhd._VP * 3)(*dp[5:]), 1) == 0
    for a, d in zip(arrays, dst):
        assert np.array_equal(a.ravel(), d.cpu().numpy())


def test_batch_primitives_of_the_changed_boxes_only():
    """CFL dt of each box after some of the states were set anew."""
    boxes = [I.random_state((9 + 5 * i, 20 - i, 4 + i), seed=i) for i in range(9)]
    b = mhd.Batch(boxes, "fp64")
    for i, q in enumerate(boxes):
        b.set_state(i, q.cell, q.face)
    want = []
    for q in boxes:
        s = mhd.Solver(q, precision="fp64")
        s.set_state(q.cell, q.face)
        want.append(s.cfl_dt())
    assert np.allclose([b.box_dt(i) for i in range(9)], want, rtol=1e-13, atol=0)
    b.step(want[0] * 0.1, 1)
    b.set_state(4, boxes[4].cell, boxes[4].face)
    assert abs(b.box_dt(4) / want[4] - 1) < 1e-13
    assert all(b.box_dt(i) != want[i] for i in range(9) if i != 4)
