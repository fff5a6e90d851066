"""The 64-bit fixed-point arithmetic of the FP64 kernels (csrc/fix64.cuh),
compiled for the host and compared with exact integers."""
import ctypes as C
import os
import subprocess
from fractions import Fraction

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    from paper_1910_01946_gb300 import _build
    cuda = os.path.join(os.path.dirname(os.path.dirname(_build.nvcc())), "include")
    so = str(tmp_path_factory.mktemp("fix64") / "fix64_host.so")
    subprocess.run(["g++", "-O1", "-std=c++17", "-fwrapv", "-shared", "-fPIC", "-I", _build.CSRC, "-I", cuda,
                    os.path.join(ROOT, "tests", "fix64_host.cpp"), "-o", so], check=True)
    return C.CDLL(so)


def split(v):
    lo = ((v + 2 ** 31) % 2 ** 32) - 2 ** 31
    return lo, (v - lo) >> 32


ROWS = {
    # integers of K whose largest is just above 2^58, 2^59 and just below 2^60
    "just above 2^58": lambda rng: rng.integers(-2 ** 58 + 1, 2 ** 58, 9),
    "just below 2^60": lambda rng: rng.integers(-2 ** 60 + 1, 2 ** 60, 9),
    "largest low words": lambda rng: rng.integers(-2 ** 26, 2 ** 26, 9) * 2 ** 32 + rng.choice([-1, 1], 9) * (2 ** 31 - 1),
    "one large entry": lambda rng: np.append(rng.integers(-2 ** 40, 2 ** 40, 8), 2 ** 58 + 12345),
}


@pytest.mark.parametrize("rows", sorted(ROWS))
@pytest.mark.parametrize("spread", [0, 20, 60])
def test_rows_of_the_tangent_product(lib, rows, spread):
    """Error bound, for a largest entry of 2^58 and a largest component of 2^55 or
    more: p is truncated by less than a unit (2^-55 per entry, nine entries),
    the dropped products of the low words are below 2^31 2^28 (2^-54 per entry),
    the sum's last bit is 2^57 (2^-56) and the result is rounded to double:
    2^-53 |row| + 7 2^-53 max|K| max|p|.  p's components differ by up to 2^spread."""
    rng = np.random.default_rng(len(rows) + spread)
    n = 400
    K = np.zeros((n, 9), dtype=object)
    words = np.zeros((n, 9, 2), dtype=np.int32)
    p = rng.uniform(-1.0, 1.0, (n, 9)) * 2.0 ** -rng.uniform(0, spread, (n, 9)) * 2.0 ** rng.integers(-80, 80, (n, 1))
    ek = rng.integers(930, 1030, n).astype(np.int32)
    for i in range(n):
        row = [int(x) for x in ROWS[rows](rng)]
        row[i % 9] = int(np.sign(row[i % 9]) or 1) * max(abs(row[i % 9]), 2 ** 58)   # the largest: 2^58 or more
        for j in range(9):
            K[i, j], words[i, j] = row[j], split(row[j])
    out = np.zeros(n)
    ptr = lambda a: a.ctypes.data_as(C.c_void_p)
    lib.rows9(n, ptr(words), ptr(ek), ptr(p), ptr(out))
    for i in range(n):
        unit = Fraction(2) ** int(ek[i] - 1016)
        exact = sum(K[i, j] * Fraction(float(p[i, j])) for j in range(9)) * unit
        big = max(abs(k) for k in K[i]) * unit * Fraction(float(np.abs(p[i]).max()))
        err = abs(Fraction(float(out[i])) - exact)
        assert err <= Fraction(1, 2 ** 53) * (abs(exact) + 7 * big), (i, float(err / big) * 2 ** 53)


def test_non_finite_and_zero_rows(lib):
    words = np.tile(np.array([123, 2 ** 27], dtype=np.int32), (3, 9, 1))
    p = np.ones((3, 9))
    p[0, 4] = np.nan
    p[1] = 0.0
    ek = np.array([970, 970, 1 << 20], dtype=np.int32)
    out = np.zeros(3)
    ptr = lambda a: a.ctypes.data_as(C.c_void_p)
    lib.rows9(3, ptr(words), ptr(ek), ptr(p), ptr(out))
    assert np.isnan(out[0]) and out[1] == 0.0 and np.isnan(out[2])


def test_values_near_the_bottom_of_the_range(lib):
    """A value of 2^-959 or more keeps 53 bits through 56-bit integers on its own
    scale, a smaller one the bits above 2^-1016; results below the normal range
    round to denormals.  K = 2^59 on the scale that makes it 1."""
    rng = np.random.default_rng(5)
    n = 2000
    p = np.zeros((n, 9))
    p[:, 4] = np.ldexp(rng.uniform(1.0, 2.0, n) * rng.choice([-1, 1], n), rng.integers(-1074, -700, n))
    words = np.zeros((n, 9, 2), dtype=np.int32)
    words[:, 4, 1] = 2 ** 27
    ek = np.full(n, 1016 - 59, dtype=np.int32)
    out = np.zeros(n)
    ptr = lambda a: a.ctypes.data_as(C.c_void_p)
    lib.rows9(n, ptr(words), ptr(ek), ptr(p), ptr(out))
    x = p[:, 4]
    assert np.all(np.abs(out - x) <= np.where(np.abs(x) >= 2.0 ** -959, 2.0 ** -53 * np.abs(x), 2.0 ** -1014))
    words[:, 4, 1] = 2 ** 27 + 2 ** 26
    ek[:] = 1016 - 59 - 200                                # 1.5 2^-200 times p
    lib.rows9(n, ptr(words), ptr(ek), ptr(p), ptr(out))
    assert np.all(np.abs(out - 1.5 * 2.0 ** -200 * x) <= 2.0 ** -52 * np.abs(out) + 2.0 ** -1074)
