"""The float64 density of LBM_MIXED_RHO64 is an integer sum of 16 float32 values (csrc/fft_fixed.cuh, sum16):
compiled for the host and compared with exact sums, over the float32 range.

Bound: the last rounding, 2^-53 of the sum, and 16 values cut off at 2^-58 of twice the largest."""
import os
import subprocess
from fractions import Fraction

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CUDA = os.environ.get("CUDA_HOME", "/usr/local/cuda")

SOURCE = r"""
#include "fft_fixed.cuh"
#include <cstdio>
int main() {  // 16 floats in; a flag and the sum's bits out
    unsigned f[16];
    unsigned long long out[2];
    while (fread(f, 4, 16, stdin) == 16) {
        out[0] = lbm::fixed::sum16(f, out[1]);
        fwrite(out, 8, 2, stdout);
    }
}
"""


@pytest.fixture(scope="module")
def sum16(tmp_path_factory):
    d = tmp_path_factory.mktemp("sum16")
    (d / "s.cpp").write_text(SOURCE)
    subprocess.run(["g++", "-std=c++17", "-O1", "-w", "-I", os.path.join(ROOT, "paper_1403_3746_gb300", "csrc"), "-I",
                    os.path.join(CUDA, "include"), "-o", str(d / "s"), str(d / "s.cpp")], check=True)

    def run(f):
        out = subprocess.run([str(d / "s")], input=np.ascontiguousarray(f, np.float32).tobytes(), capture_output=True, check=True)
        raw = np.frombuffer(out.stdout, np.uint64).reshape(-1, 2)
        return raw[:, 0] != 0, raw[:, 1].view(np.float64)

    return run


def test_sum_at_any_magnitude(sum16):
    rng = np.random.default_rng(3)
    rows = []
    for e in range(-62, 126, 2):  # the largest of a row within [2^e, 2^(e + 1)), others as large or far smaller
        spread = np.repeat([1, 4, 40, 70], 10)[:, None]
        r = np.ldexp(rng.uniform(-1, 1, (40, 16)), e - rng.integers(0, spread, (40, 16)))
        r[:, 5] = np.ldexp(rng.uniform(1, 2, 40), e) * rng.choice([-1, 1], 40)
        rows.append(r)
    rows.append(np.full((1, 16), 1e-10) * np.arange(1, 17))
    f = np.concatenate(rows).astype(np.float32)
    f[::7, 3] = 0.0
    ok, s = sum16(f)
    assert ok.all()
    for row, got in zip(f.astype(np.float64), s):
        want = sum(map(Fraction, row.tolist()))
        assert abs(Fraction(got) - want) <= abs(want) / 2 ** 53 + Fraction(np.abs(row).max()) / 2 ** 53, (row, got, float(want))


def test_equal_and_short_values_are_exact(sum16):
    f = np.concatenate([np.ldexp(np.full((1, 16), 0.75), e) for e in range(-62, 124)]).astype(np.float32)
    ok, s = sum16(f)
    assert ok.all() and np.array_equal(s, 16 * f[:, 0].astype(np.float64))


@pytest.mark.parametrize("value", [0.0, 1e-30, np.inf, -np.inf, np.nan])
def test_values_left_to_the_float64_sum(sum16, value):
    f = np.zeros((1, 16), np.float32)
    f[0, 4] = value
    assert not sum16(f)[0][0]
