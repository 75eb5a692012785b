"""lbm_moments with targets that are device memory: the same answer below the size that is read through one
host buffer as above it (that buffer's contents are never stored through such a pointer)."""
import ctypes

import numpy as np
import pytest

import paper_1403_3746_gb300 as lbm
import synthetic

pytestmark = pytest.mark.gpu


def read_into_device(nx, ny):
    import torch
    with lbm.Simulation(nx, ny, lbm.default_params()) as s:
        s.init(*synthetic.spinodal(nx, ny, 1.0, 0.01, 0.9, seed=6))
        ref = s.moments()
        t = torch.zeros((4, ny, nx), dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        rc = lbm.lib().lbm_moments(s._h, *[ctypes.cast(ctypes.c_void_p(t[j].data_ptr()), ctypes.POINTER(ctypes.c_double))
                                           for j in range(4)])
        if rc == 0:
            torch.cuda.synchronize()
            assert all(np.array_equal(t[j].cpu().numpy(), ref[j]) for j in range(4))
        assert all(np.array_equal(a, b) for a, b in zip(s.moments(), ref))
        return rc


def test_device_targets_at_any_size():
    assert read_into_device(16, 2) == read_into_device(32, 32) == read_into_device(256, 256)
