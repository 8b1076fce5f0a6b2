"""div_known (csrc/known_divisor.cuh), the FP64 tables' division by a number
whose reciprocal is known, against the division it stands for.  Compiled for
the host: its operations are IEEE, the same as on the device."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

from paper_2405_04229_gb300 import build


@pytest.fixture(scope="module")
def div_known(tmp_path_factory):
    d = str(tmp_path_factory.mktemp("div"))
    src, so = os.path.join(d, "d.cpp"), os.path.join(d, "d.so")
    with open(src, "w") as f:
        f.write('#define __host__\n#define __device__\n#include "known_divisor.cuh"\n'
                'extern "C" void run(const double* x, const double* c, long n, double* out) {\n'
                '    for (long i = 0; i < n; ++i) out[i] = cs::div_known(x[i], c[i], 1.0 / c[i]);\n}\n')
    subprocess.run(["g++", "-O2", "-ffp-contract=off", "-shared", "-fPIC", "-I", build.CSRC, src, "-o", so], check=True)
    L = C.CDLL(so)

    def f(x, c):
        x, c = np.broadcast_arrays(x, c)
        x, c = np.ascontiguousarray(x, np.float64), np.ascontiguousarray(c, np.float64)
        out = np.empty(x.shape)
        L.run(x.ctypes.data_as(C.c_void_p), c.ctypes.data_as(C.c_void_p), C.c_long(x.size), out.ctypes.data_as(C.c_void_p))
        return out
    return f


def _mantissas(rng, n):
    """Random ones, and the fewest and the most bits set."""
    m = rng.uniform(1.0, 2.0, n)
    k = rng.integers(0, 52, n)
    pick = rng.integers(0, 4, n)
    m = np.where(pick == 1, 1.0 + np.ldexp(1.0, -k - 1), m)
    return np.where(pick == 2, 2.0 - np.ldexp(1.0, -k - 1), m)


@pytest.mark.parametrize("e_c", [(-14, 1), (9, 31), (-600, 600)])   # roots q, scale heights [m, cm], any
def test_same_rounding_as_the_division(div_known, e_c):
    rng = np.random.default_rng(e_c[1])
    n = 2_000_000
    c = np.ldexp(_mantissas(rng, n), rng.integers(*e_c, n))
    x = np.ldexp(_mantissas(rng, n), rng.integers(-959, 960, n)) * rng.choice([-1.0, 1.0], n)
    with np.errstate(over="ignore", under="ignore"):
        q = x / c
    ok = (np.abs(q) >= 2.0**-1000) & (np.abs(q) < 2.0**1000)
    assert ok.sum() > n // 4
    assert np.array_equal(div_known(x, c)[ok], q[ok])


def test_zero_and_equal_operands(div_known):
    c = np.ldexp(_mantissas(np.random.default_rng(1), 100_000), 3)
    assert np.all(div_known(0.0 * c, c) == 0.0)
    assert np.all(div_known(c, c) == 1.0)


def test_two_ulps_where_the_remainder_underflows(div_known):
    """The remainder is then rounded to a multiple of 2^-1074, at most 2^-1075 off: an ulp of a quotient
    of a normal x; half an ulp more for rounding the sum, and another half for the division's own."""
    rng = np.random.default_rng(5)
    n = 1_000_000
    c = np.ldexp(_mantissas(rng, n), rng.integers(-14, 0, n))
    x = np.ldexp(_mantissas(rng, n), rng.integers(-1022, -960, n))
    q = x / c
    assert np.all(np.abs(div_known(x, c) - q) <= 2.0 * np.spacing(q))
