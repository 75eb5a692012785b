"""The float64 path's line transforms run in 64-bit fixed point with one exponent per line
(csrc/fft_fixed.cuh). Checked through advection-only Euler steps, f_i - dt v_i . grad f_i, on every
line length along both axes, for lines with a large mean, sparse lines, noise and zero lines.

Bound. Per pair of lines with largest magnitude A (two fields of a row, or two neighbouring
columns of a field, share a complex line and its exponent) the points are rounded at 2^-54 A or
finer and the passes at no more than 2^-46 A over sqrt(N), so with the axis's largest multiplier d
an entry of the derivative is within 2^-47 A d; numpy's float64 transforms, the reference, get as
much again, and the sums of the result two roundings.
"""
import numpy as np
import pytest

import paper_1403_3746_gb300 as lbm
from oracle.dvm import D2V16
from oracle.wfft import dft_indices, keff, spectral_deriv

pytestmark = pytest.mark.gpu

FLAGS = lbm.LBM_FLAG_NO_COLLISION | lbm.LBM_FLAG_NO_FORCE | lbm.LBM_FLAG_EULER
ROW_PARTNER = [2, 1, 0, 3, 6, 5, 4, 7, 9, 8, 11, 10, 13, 12, 15, 14]  # opposite v_x, same complex line


def lines(n, rng):
    x = np.arange(n)
    bump = 1.0 / np.cosh(np.minimum(np.abs(x - n / 3), 300.0) / 2) ** 2
    spike = np.zeros(n)
    spike[n // 2] = 1.0
    return [np.ones(n), np.zeros(n), 1 + 0.01 * rng.uniform(-1, 1, n), rng.uniform(-1, 1, n), bump * 1e-3, spike,
            0.3 + 1.5 * bump, 1e-17 * rng.uniform(-1, 1, n), np.sin(2 * np.pi * x / n) + 2, -bump, 1e3 * spike,
            np.where(x < n / 2, 1.8, 0.32), rng.uniform(0, 1, n), bump - 1, np.cos(np.pi * x), -np.ones(n)]


@pytest.mark.parametrize("axis", [0, 1])
@pytest.mark.parametrize("log2n", range(1, 13))
def test_line_derivative_every_length(log2n, axis):
    n, other = 1 << log2n, 4
    rng = np.random.default_rng(100 * log2n + axis)
    # one kind of line per field; neighbouring lines differ by a factor, so that a mixed-up one shows
    f = np.stack(lines(n, rng))[:, None, :] * np.array([1.0, -0.5, 0.25, 0.75])[None, :, None]
    if axis == 0:
        f = np.swapaxes(f, 1, 2)
    f = np.ascontiguousarray(f)
    ny, nx = f.shape[1:]
    d = D2V16()
    A = np.abs(f).max(axis=(1, 2))
    Ax = np.maximum(A, A[ROW_PARTNER])
    dx, dy = (float(np.abs(keff(dft_indices(k), k, 1.0)).max()) for k in (nx, ny))
    expect, bound = f.copy(), 2.0 ** -51 * A
    for i in range(16):
        expect[i] -= d.vx[i] * spectral_deriv(f[i], 1, 0, 1.0, 1.0) + d.vy[i] * spectral_deriv(f[i], 0, 1, 1.0, 1.0)
        bound[i] += (2.0 ** -46 + 2.0 ** -51) * (abs(d.vx[i]) * dx * Ax[i] + abs(d.vy[i]) * dy * A[i])
    with lbm.Simulation(nx, ny, lbm.default_params(flags=FLAGS, dt=1.0, tau=1.0, dx=1.0, dy=1.0)) as s:
        s.init(np.ones((ny, nx)), *[np.zeros((ny, nx))] * 2, np.ones((ny, nx)))
        s.set_f(f)
        s.step(1)
        got = s.get_f()
    err = np.abs(got - expect).max(axis=(1, 2))
    assert np.all(err <= bound), (log2n, axis, err, bound)


@pytest.mark.parametrize("power", [-900, -300, 300, 900])
def test_line_derivative_scales_exactly_with_powers_of_two(power):
    """A common exponent per line: dense lines scaled by 2^p give the result scaled by 2^p, bit for
    bit, over the whole float64 range (outside the float32 range as well)."""
    rng = np.random.default_rng(7)
    nx, ny = 128, 64
    f = 1 + 0.1 * rng.uniform(-1, 1, (16, ny, nx))
    out = []
    for p in (0, power):
        with lbm.Simulation(nx, ny, lbm.default_params(flags=FLAGS, dt=1e-3, tau=1.0, dx=1.0, dy=1.0)) as s:
            s.init(np.ones((ny, nx)), *[np.zeros((ny, nx))] * 2, np.ones((ny, nx)))
            s.set_f(np.ldexp(f, p))
            s.step(1)
            out.append(np.ldexp(s.get_f(), -p))
    assert np.array_equal(out[0], out[1])
