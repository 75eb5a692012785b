"""Accuracy of the float64 path's fixed-point line derivatives (csrc/fft_line.cuh) by kind of line, against
80-bit (or wider) sums: no worse than twice numpy's float64 transforms on the same lines.

Read off advection-only Euler steps f_i - dt v_i . grad f_i with a step so large (2^60) that their
rounding is the derivative's. Fields are constant along the other axis, or take two lines in turn there (the mean and the
Nyquist index of four points), so its derivative is exactly zero.

Bound of the root-mean-square error: twice numpy's, and 12 2^-53 of the derivative's for what has nothing
to do with the transform: the multiplier table (a series of eight terms in float64, about 10 roundings),
the factor dt v_i and the final rounding. A host restatement of the passes against __float128 sums gives
0.00 to 1.0 times the error of a float64 transform by the same passes for these kinds, 4 to 4096 points,
and numpy's transforms have 0.5 to 1 times that error. Kinds whose sums float64 holds exactly (few-bit
values) are left out at 4096 points, where the restatement gives 1.4.
"""
import numpy as np
import pytest

import paper_1403_3746_gb300 as lbm
from oracle.dvm import D2V16

pytestmark = pytest.mark.gpu

FLAGS = lbm.LBM_FLAG_NO_COLLISION | lbm.LBM_FLAG_NO_FORCE | lbm.LBM_FLAG_EULER
PAIRS = [(0, 2), (4, 6), (8, 9), (10, 11), (12, 13), (14, 15)]  # fields whose rows share a complex line
COLUMNS = [1, 3, 5, 7, 8, 9, 10, 11, 12, 13, 14, 15]  # fields that move along y
LD = np.longdouble


def kinds(n, rng):
    """Pairs of lines."""
    x = np.arange(n)
    u = lambda: rng.uniform(-1, 1, n)
    drop = 0.32 + 1.48 * 0.5 * (1 + np.tanh((n / 4 - np.abs(x - n / 2)) / 2))
    bump = np.exp(-((x - n // 3) / 2.0) ** 2)
    point = (x == n // 3).astype(float)
    return {
        "noise": (u(), u()),
        "noise about a mean": (1 + 0.01 * u(), 0.3 + 0.003 * u()),
        "smooth": (1 + 0.5 * np.sin(2 * np.pi * x / n), 0.9 + 0.2 * np.cos(4 * np.pi * x / n)),
        "droplet beside a constant": (drop, np.full(n, 0.85)),
        "two sharp levels beside a constant": (np.where(x < n // 2, 1.045, 0.955), np.full(n, 0.9975)),
        "two far levels beside a constant": (np.where(x < n // 2, 1.8123456789, 0.3212345678), np.full(n, 0.9)),
        "constant but for one point": (0.9 + 0.2 * point, np.full(n, 0.85)),
        "few points wide": (0.9 + 0.2 * bump, np.full(n, 0.85)),
        "constant to 1e-4": (1 + 1e-4 * u(), 0.9 + 1e-4 * u()),
        "constant to 1e-8": (1 + 1e-8 * u(), 0.9 + 1e-8 * u()),
        "points alone": (point, -0.7 * np.roll(point, 5)),
        "few bits": (1 + 0.5 * point, np.ones(n)),
    }


def multiplier(n, dtype):
    """The spectral derivative's multipliers (eight terms, dx = 1), indices 0 .. n/2."""
    pi = dtype(np.arccos(LD(-1)))
    phi = np.sin(pi * np.arange(n // 2 + 1).astype(dtype) / dtype(n))
    c = [(1, 1), (1, 6), (3, 40), (5, 112), (35, 1152), (63, 2816), (231, 13312), (143, 10240)]
    k = dtype(2) * sum(dtype(a) / dtype(b) * phi ** (2 * j + 1) for j, (a, b) in enumerate(c))
    k[-1] = 0
    return k


def exact(lines, n, where):
    """d/dx at the given points by direct sums in long double."""
    k = multiplier(n, LD)
    s = np.sin(2 * LD(np.arccos(LD(-1))) * np.arange(n).astype(LD) / LD(n))
    j = np.arange(n)
    col = np.array([-2 * np.sum(k[1:n // 2] * s[(r * np.arange(1, n // 2)) % n]) for r in range(n)], dtype=LD) / n
    h = np.asarray(lines).astype(LD)
    return np.stack([h @ col[(r - j) % n] for r in where], axis=1)


def difference(f, dt):
    """f - f after one advection-only Euler step."""
    ny, nx = f.shape[1:]
    with lbm.Simulation(nx, ny, lbm.default_params(flags=FLAGS, dt=dt, tau=1.0, dx=1.0, dy=1.0)) as s:
        s.init(np.ones((ny, nx)), *[np.zeros((ny, nx))] * 2, np.ones((ny, nx)))
        s.set_f(f)
        s.step(1)
        return f.astype(LD) - s.get_f()


@pytest.mark.parametrize("log2n", [2, 3, 4, 5, 6, 8, 9, 10, 12])
def test_line_derivative_error_by_kind_of_line(log2n):
    n, dt, d = 1 << log2n, 2.0 ** 60, D2V16()
    by_kind = kinds(n, np.random.default_rng(log2n))
    if log2n == 12:
        by_kind.pop("few bits")
    names = list(by_kind)
    flat = [line for name in names for line in by_kind[name]]
    where = np.arange(n) if n <= 512 else np.unique(np.r_[:16, n // 3 - 64:n // 3 + 64, n // 2 - 32:n // 2 + 32, n - 16:n])
    truth = exact(flat, n, where)
    plain = np.fft.irfft(1j * multiplier(n, np.float64) * np.fft.rfft(np.array(flat), axis=1), n, axis=1)[:, where]
    rms = lambda e: np.sqrt(np.sum(np.asarray(e, dtype=LD) ** 2, axis=1)).astype(float)
    bound = 2 * rms(plain - truth) + 12 * 2.0 ** -53 * rms(truth)
    # a pair's bound is that of its two lines together: they share a complex line
    bound = np.hypot(bound[0::2], bound[1::2])
    got = []  # per axis and kind: its two lines' derivatives
    for first in range(0, len(names), len(PAIRS)):  # rows
        f = np.ones((16, 4, n))
        for name, (a, b) in zip(names[first:], PAIRS):
            f[a], f[b] = by_kind[name][0][None, :], by_kind[name][1][None, :]
        out = difference(f, dt)
        got += [("rows", p, [out[i][1][where] / (dt * d.vx[i]) for i in PAIRS[p - first]])
                for p in range(first, min(first + len(PAIRS), len(names)))]
    f = np.ones((16, n, 4))  # columns, the two lines in turn
    for p, i in enumerate(COLUMNS[:len(names)]):
        f[i] = np.stack([by_kind[names[p]][c & 1] for c in range(4)], axis=1)
    out = difference(f, dt)
    got += [("columns", p, [out[i][where, c] / (dt * d.vy[i]) for c in (0, 1)]) for p, i in enumerate(COLUMNS[:len(names)])]
    for axis, p, lines in got:
        err = np.hypot(*rms(np.asarray(lines, dtype=LD) - truth[2 * p:2 * p + 2]))
        assert err <= bound[p], (n, axis, names[p], err, bound[p])


@pytest.mark.parametrize("axis", [0, 1])
@pytest.mark.parametrize("log2n", [3, 6, 8, 10])
def test_small_line_beside_a_large_one(log2n, axis):
    """The two lines of a complex line have exponents of their own: one 1e-9 times the other (a dilute density
    beside the temperature) keeps its accuracy. The bound is each line's own as above, and its partner's
    at the same scale, which the transform may leave in it."""
    n, dt, d = 1 << log2n, 2.0 ** 60, D2V16()
    x = np.arange(n)
    lines = np.array([1e-9 * (1 + 0.2 * np.sin(2 * np.pi * x / n)), 0.9 + 1e-3 * np.cos(2 * np.pi * x / n)])
    where = np.arange(n) if n <= 512 else np.r_[:200]
    truth = exact(lines, n, where)
    plain = np.fft.irfft(1j * multiplier(n, np.float64) * np.fft.rfft(lines, axis=1), n, axis=1)[:, where]
    rms = lambda e: np.sqrt(np.sum(np.asarray(e, dtype=LD) ** 2, axis=1)).astype(float)
    own = 2 * rms(plain - truth) + 12 * 2.0 ** -53 * rms(truth)
    top = np.abs(lines).max(axis=1)
    bound = own + own[::-1] * top / top[::-1]
    f = np.ones((16, 4, n))
    if axis == 0:
        f[0], f[2] = lines[0], lines[1]
        out = difference(f, dt)
        got = [out[0][1][where] / (dt * d.vx[0]), out[2][1][where] / (dt * d.vx[2])]
    else:
        f[1] = lines[[0, 1, 0, 1]]
        out = difference(np.ascontiguousarray(np.swapaxes(f, 1, 2)), dt)
        got = [out[1][where, c] / (dt * d.vy[1]) for c in (0, 1)]
    assert np.all(rms(np.asarray(got) - truth) <= bound)
