"""Grids of two rows: a 2-point axis has only the mean and the Nyquist index, whose derivative
multipliers are zero, so the library runs no column pass there. The y-derivative fields must stay
zero whatever ran on the handle before."""
import numpy as np
import pytest

import oracle
import paper_1403_3746_gb300 as lbm
import synthetic
from oracle.dvm import D2V16
from oracle.model import init_feq, rk2_step

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,tol", [(lbm.LBM_FP64, 1e-12), (lbm.LBM_MIXED, 2e-6), (lbm.LBM_MIXED_RHO64, 2e-6)])
def test_two_rows_after_a_state_that_blew_up(precision, tol):
    # a non-finite state, its diagnostics (which differentiate along y), then a new start: the run
    # must be that of a fresh handle, and the oracle's (tolerances: those of the parity tests)
    nx, ny, steps = 256, 2, 5
    fields = synthetic.slab(nx, ny, 1.4, 0.6, 0.95, noise=1e-3, seed=11)
    with lbm.Simulation(nx, ny, lbm.default_params(precision=precision)) as s:
        s.init(*fields)
        f = s.get_f()
        s.set_f(f * 1e30)
        s.step(3)
        with pytest.raises(lbm.LbmError):
            s.diagnostics()
        s.init(*fields)
        s.step(steps)
        got, diag = s.get_f(), s.diagnostics()
    with lbm.Simulation(nx, ny, lbm.default_params(precision=precision)) as s:
        s.init(*fields)
        s.step(steps)
        assert np.array_equal(got, s.get_f())
    p, d = oracle.Params(), D2V16(oracle.Params().eta0)
    fo = init_feq(d, *fields, p)
    for _ in range(steps):
        fo = rk2_step(d, fo, p)
    assert np.max(np.abs(got - fo)) <= tol * np.max(np.abs(fo))
    assert abs(diag["mass"] / (oracle.moments(d, fo, p.b)[0].sum() * p.dx * p.dy) - 1) <= max(tol, 1e-12)
