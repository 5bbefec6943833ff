"""The fixed-point line transforms compiled for the host, at the bound of their
scale: lines that one to three cells dominate, at every leg of the first
butterfly, over the mantissas and phases that bring a value close to it."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_2405_02603_gb300 import build as B

# Outputs are sums of modulus <= the line's 1-norm, rounded once to doubles
# (2^-53 of it).  The line is held in units of at most 2^-60.4 of it, 256 times
# that after the five stages of the longest schedule.  With up to three cells
# the first stage is off by at most 4.5 units, and a later one's sum of R takes
# over a quarter of that of each input and a rounding: below 40 units with
# three stages of 8 (2^-51 of the norm), 5 with 5, 5, 3, 3, 2 (2^-50.1).
TOL = 8 * 2.0 ** -53
PI = np.longdouble("3.14159265358979323846264338327950288")
AMPS = [1.0, 1.1, 1.25, 1.4, 1.6, 1.8]


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    here = os.path.dirname(os.path.abspath(__file__))
    out = str(tmp_path_factory.mktemp("fx") / "fx_line_host.so")
    cmd = [B.nvcc()] + B.ARCH + ["-O1", "-std=c++17", "--expt-relaxed-constexpr", "-diag-suppress", "20093", "-Xcompiler",
                                 "-fPIC", "-shared", "-I", os.path.join(B.ROOT, "include"), "-I",
                                 B.CSRC, os.path.join(here, "host", "fx_line_host.cu"), "-o", out]
    subprocess.run(cmd, check=True)
    return ctypes.CDLL(out)


def sparse_lines(n, n_in, cells, count, rng):
    """(positions, values): `count` lines, the first cell at every position."""
    pos = rng.integers(0, n_in, size=(count, cells))
    pos[:, 0] = np.arange(count) % n_in
    amp = np.array(AMPS)[rng.integers(0, len(AMPS), size=(count, cells))]
    amp[:, 1:] *= 2.0 ** -rng.integers(0, 12, size=(count, cells - 1))
    return pos, amp * np.exp(2j * np.pi * rng.uniform(size=(count, cells)))


def check(fn, n, n_in, sign, cells, rng):
    count = max(2 * n_in, 512)
    pos, val = sparse_lines(n, n_in, cells, count, rng)
    x = np.zeros((count, n), np.complex128)
    want = np.zeros((count, n), np.clongdouble)
    k = np.arange(n)
    w = np.exp(sign * 2j * PI * k.astype(np.longdouble) / n)
    for c in range(cells):
        np.add.at(x, (np.arange(count), pos[:, c]), val[:, c])
        want += val[:, c, None] * w[(pos[:, c, None] * k) % n]
    got = np.full_like(x, np.nan)
    assert fn(n, sign, count, x.ctypes.data_as(ctypes.c_void_p), got.ctypes.data_as(ctypes.c_void_p)) == 0
    norm = np.abs(val).sum(1)
    err = np.abs(got - want).max(1) / norm
    print("n=%d sign=%d cells=%d: %.2e" % (n, sign, cells, err.max()))
    assert err.max() <= TOL, (err > TOL).mean()


@pytest.mark.parametrize("n", [64, 96, 128, 192, 256, 384, 512, 1024])
@pytest.mark.parametrize("sign", [-1, 1])
def test_specialised_shapes(lib, n, sign):
    rng = np.random.default_rng(n + sign)
    for cells in (1, 2, 3):
        check(lib.fx_lines, n, n // 2 if sign < 0 else n, sign, cells, rng)


@pytest.mark.parametrize("n", [2, 3, 5, 8, 9, 15, 25, 32, 60, 90, 100, 150, 200, 240, 250, 450, 625])
@pytest.mark.parametrize("sign", [-1, 1])
def test_generic_schedules(lib, n, sign):
    rng = np.random.default_rng(n + sign)
    for cells in (1, 2, 3):
        check(lib.fx_lines_generic, n, n, sign, cells, rng)
