"""Device arrays that end before the state does: the copy kernel must not
read or write past their allocation.  Such calls are refused with
MHD_ERR_CUDA before anything runs on the GPU, as the runtime's copy refuses
them, wherever the allocation's end is known."""
import ctypes

import numpy as np
import pytest

from paper_2606_12753_gb300 import inputs as I
from paper_2606_12753_gb300 import mhd

pytestmark = pytest.mark.gpu


def _allocation(ptr):
    """(bytes from ptr to the end of its allocation, whether it is one cudaMalloc)."""
    cuda = ctypes.CDLL("libcuda.so.1")
    start, size, whole = ctypes.c_ulonglong(), ctypes.c_size_t(), ctypes.c_uint()
    for what, out in ((11, start), (12, size), (10, whole)):   # RANGE_START_ADDR, RANGE_SIZE, LEGACY_CUDA_IPC_CAPABLE
        if cuda.cuPointerGetAttribute(ctypes.byref(out), what, ctypes.c_ulonglong(ptr)) != 0:
            return 0, False
    return start.value + size.value - ptr, bool(whole.value)


@pytest.mark.parametrize("short", [0, 4, 5, 7])
def test_arrays_that_end_early_are_refused(short):
    import torch
    box = I.uniform_state((128, 64, 64))
    want = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in list(box.cell) + list(box.face)]
    arrays = [w.clone() for w in want]
    torch.cuda.empty_cache()
    few = torch.zeros(64, dtype=torch.float64, device="cuda")    # in an allocation of 2 MiB
    left, whole = _allocation(few.data_ptr())
    if not whole or left >= 8 * box.ncell:
        pytest.skip("the end of this allocation is not known to the library")
    p = [a.data_ptr() for a in arrays]
    s = mhd.Solver(box, precision="fp64")
    mhd.mhd_set_state(s.h, p[:5], p[5:], 1)
    bad = list(p)
    bad[short] = few.data_ptr()
    for call in (mhd.mhd_set_state, mhd.mhd_get_state):
        with pytest.raises(mhd.MHDError) as ei:
            call(s.h, bad[:5], bad[5:], 1)
        assert ei.value.code == mhd.MHD_ERR_CUDA
    for a in arrays:
        a.fill_(-1.0)
    mhd.mhd_get_state(s.h, p[:5], p[5:], 1)     # the handle stays usable, its state unchanged
    for a, w in zip(arrays, want):
        assert torch.equal(a, w)
    assert float(few.abs().sum()) == 0.0


def test_an_array_that_ends_with_its_allocation_is_taken():
    import torch
    n = (64, 64, 64)                            # 2 MiB of FP64, one allocation each
    box = I.random_state(n, seed=2)
    want = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in list(box.cell) + list(box.face)]
    p = [a.data_ptr() for a in want]
    s = mhd.Solver(box, precision="fp64")
    mhd.mhd_set_state(s.h, p[:5], p[5:], 1)
    out = [torch.zeros_like(a) for a in want]
    q = [a.data_ptr() for a in out]
    mhd.mhd_get_state(s.h, q[:5], q[5:], 1)
    for a, w in zip(out, want):
        assert torch.equal(a, w)
