"""A training step by one call against its three parts."""
import numpy as np
import pytest


@pytest.mark.gpu
@pytest.mark.parametrize("n", [1, 127, 128])
def test_one_call_equals_its_parts(n):
    """One 128-row tile at most: its sums have one order, so every number is the same."""
    import torch
    from paper_2606_12753_gb300 import mhd, switch_train
    x = torch.from_numpy(np.random.default_rng(n).standard_normal((n, 16)).astype(np.float32)).cuda()
    y = (x[:, 0] > 0).float()
    one, parts = (switch_train.Switch(switch_train.he_init(2)) for _ in range(2))
    for t in (1, 2):
        one.step(x, y, 1e-3)
        parts.g.zero_()
        mhd.mlp_backward(parts.block.data_ptr(), x.data_ptr(), y.data_ptr(), n, parts.g.data_ptr())
        mhd.mlp_adam(parts.block.data_ptr(), parts.m.data_ptr(), parts.v.data_ptr(), parts.g.data_ptr(), t, lr=1e-3)
    torch.cuda.synchronize()
    assert one.t == 2
    for a, b in ((one.block, parts.block), (one.m, parts.m), (one.v, parts.v), (one.g, parts.g)):
        assert torch.equal(a, b)


@pytest.mark.gpu
def test_refused_rows_leave_the_step_count():
    import torch
    from paper_2606_12753_gb300 import mhd, switch_train
    sw = switch_train.Switch(switch_train.he_init(2))
    x = torch.zeros(16 * 8 + 1, device="cuda")[1:].view(8, 16)   # rows off their 16-byte boundary
    before = sw.block.clone()
    with pytest.raises(mhd.MHDError) as ei:
        sw.step(x, torch.zeros(8, device="cuda"), 1e-3)
    assert ei.value.code == mhd.MHD_ERR_INVALID and sw.t == 0 and torch.equal(sw.block, before)
