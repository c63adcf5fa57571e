"""The FP64 learned switch takes its default z-chunk length from the box's
size, so neither its states nor its per-face choices and logits may depend on
the length."""
import numpy as np
import pytest

from paper_2606_12753_gb300 import inputs as I
from paper_2606_12753_gb300 import mhd, switch_train

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims", [(24, 24, 24), (64, 40, 50), (33, 70, 3)])
def test_chunk_length_leaves_the_learned_bits(dims):
    import torch
    box = I.random_state(dims, seed=5)
    sw = switch_train.Switch(switch_train.he_init(3))
    got = []
    for tz in (0, 1, 7, 32, dims[2]):
        s = mhd.Solver(box, precision="fp64", riemann="learned", tile=(0, 0, tz))
        s.set_switch(sw.block.data_ptr(), 0.5)
        s.set_state(box.cell, box.face)
        ch = torch.zeros(3 * box.ncell, dtype=torch.uint8, device="cuda")
        z = torch.zeros(3 * box.ncell, dtype=torch.float32, device="cuda")
        s.switch_choices(ch.data_ptr(), z.data_ptr())
        s.step(-1.0, 2)
        c, f = s.get_state()
        got.append([c] + f + [ch.cpu().numpy(), z.cpu().numpy()])
        s.close()
    assert 0.02 < got[0][4].mean() < 0.98
    for other in got[1:]:
        for a, b in zip(got[0], other):
            assert np.array_equal(a, b)
