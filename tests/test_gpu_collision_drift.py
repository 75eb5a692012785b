"""Mass and energy under the collision alone (LBM_FP64): the node's update takes f^eq from coefficients that are
the same in every step, so an error of theirs adds up step by step.

Bound: 1e-16 of mass and energy per step, mean over the nodes. The coefficients rounded once each take 2e-17 of
the energy and 3e-17 of the mass per step (mean over T = 0.8 .. 1 at rest, from the coefficients and exact ones);
the rest is for what the nodes' own roundings, which differ in sign from node to node, leave in the mean."""
import numpy as np
import pytest

import paper_1403_3746_gb300 as lbm

pytestmark = pytest.mark.gpu


def test_collision_keeps_mass_and_energy():
    n, steps = 64, 500
    rng = np.random.default_rng(5)
    rho, T = 1 + 0.5 * rng.uniform(-1, 1, (n, n)), rng.uniform(0.8, 1.0, (n, n))
    psi = np.array([7.25] * 4 + [36.0] * 4 + [2.0] * 4 + [4.5] * 4, dtype=np.longdouble)
    flags = lbm.LBM_FLAG_NO_ADVECTION | lbm.LBM_FLAG_NO_FORCE
    with lbm.Simulation(n, n, lbm.default_params(flags=flags)) as s:
        s.init(rho, np.zeros((n, n)), np.zeros((n, n)), T)
        f0 = s.get_f().astype(np.longdouble)
        s.step(steps)
        f1 = s.get_f().astype(np.longdouble)
    for w in (np.ones(16, dtype=np.longdouble), psi):
        a, b = (np.tensordot(w, f, 1).sum() for f in (f0, f1))
        assert abs(float(b / a - 1)) <= 1e-16 * steps
