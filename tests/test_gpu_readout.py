"""Moment read-out into the caller's host arrays: new ones, parts of one array, and arrays that are
pinned one by one (which may follow one another in the address space without being one allocation),
below and above the size that goes through one copy."""
import numpy as np
import pytest

import paper_1403_3746_gb300 as lbm
import synthetic

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny", [(16, 2), (64, 32), (128, 64), (256, 256), (1024, 1024)])
@pytest.mark.parametrize("precision", [lbm.LBM_FP64, lbm.LBM_MIXED])
def test_moments_into_any_host_arrays(nx, ny, precision):
    import torch
    with lbm.Simulation(nx, ny, lbm.default_params(precision=precision)) as s:
        s.init(*synthetic.spinodal(nx, ny, 1.0, 0.01, 0.9, seed=6))
        s.step(2)
        dev = [torch.empty((ny, nx), dtype=torch.float64, device="cuda") for _ in range(4)]
        s.moments_device(*dev)
        torch.cuda.synchronize()
        ref = [d.cpu().numpy() for d in dev]
        pinned = [torch.empty((ny, nx), dtype=torch.float64, pin_memory=True) for _ in range(4)]
        one = torch.empty((4, ny, nx), dtype=torch.float64, pin_memory=True).numpy()
        for out in (None, [p.numpy() for p in pinned], list(one), list(np.empty((4, ny, nx)))):
            got = s.moments(out=out)
            assert all(np.array_equal(g, r) for g, r in zip(got, ref))
