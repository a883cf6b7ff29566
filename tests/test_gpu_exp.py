"""exp_rounded of the FP64 path against exp in 60 decimal digits, rounded once: bit for bit, over
every entry of its table, both sides of the boundaries of its argument reduction, both ends
of its range and beyond, tiny arguments, and arguments whose result lies so close to the middle
of two doubles (within 2^-78) that its rounding test leaves the decision to exp_cr."""
import ctypes
import decimal
import math
import os
import subprocess

import numpy as np
import pytest

from paper_1008_2865_gb300 import build as lbbuild

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("exp") / "exp_check.so")
    subprocess.run([lbbuild._nvcc(), *lbbuild.ARCH, "-O3", "-std=c++17", "--fmad=false", "-shared",
                    "-Xcompiler", "-fPIC,-ffp-contract=off", "-I" + lbbuild.INCLUDE,
                    "-I" + lbbuild.CSRC, os.path.join(ROOT, "tests", "c", "exp_check.cu"), "-o", so],
                   check=True)
    return ctypes.CDLL(so)


def _check(lib, xs):
    x = np.array(xs, dtype=np.float64)
    y, z = np.empty_like(x), np.empty_like(x)
    ptr = [ctypes.c_void_p(v.ctypes.data) for v in (x, y, z)]
    assert lib.exp_check(*ptr, ctypes.c_int(len(x))) == 0
    with decimal.localcontext() as ctx:
        ctx.prec = 60
        want = np.array([float(decimal.Decimal(float(v)).exp()) for v in x])
    bad = np.nonzero((y != want) | (z != want))[0]
    assert len(bad) == 0, [(x[i].hex(), y[i].hex(), z[i].hex(), want[i].hex()) for i in bad[:5]]


def _around(v):
    v = float(v)
    return [np.nextafter(v, -np.inf), v, np.nextafter(v, np.inf)]


def test_every_table_entry_and_reduction_boundary(lib):
    """x = (256 m + j) ln2 / 256 and (256 m + j + 1/2) ln2 / 256 for all j."""
    xs = []
    for m in (-46, -17, -3, -1, 0, 1, 20, 45):
        for j in range(256):
            for half in (0.0, 0.5):
                xs += _around((256 * m + j + half) * math.log(2.0) / 256)
    _check(lib, [v for v in xs if abs(v) < 32.0])


def test_over_the_range(lib):
    rng = np.random.default_rng(5)
    xs = list(-rng.uniform(0.0, 4.0, 4000)) + list(rng.uniform(-32.0, 32.0, 4000))
    xs += list(rng.uniform(-700.0, 700.0, 1000))                 # beyond 32: exp_cr
    for v in (32.0, -32.0):
        xs += _around(v)
    _check(lib, xs)


def test_tiny_arguments(lib):
    """Powers of two of either sign down to the least denormal, and zero. (Not 2^-53 itself:
    its exp lies 2^-107 from the middle of two doubles, closer than exp_cr's 2^-100.)"""
    xs = [s * 2.0 ** -k for k in range(1, 1075) for s in (1.0, -1.0) if (s, k) != (1.0, 53)]
    _check(lib, xs + [0.0, -0.0])


def test_arguments_that_leave_the_rounding_open(lib):
    """exp(x) = 1 + x + x^2/2 + .. with x an odd multiple of half an ulp of the result lies
    x^2/2 from the middle of two doubles: 2^-99 .. 2^-79 for the multiples here."""
    rng = np.random.default_rng(6)
    odd = 2 * np.unique(rng.integers(8, 1 << 13, 3000)) + 1
    _check(lib, list(odd * 2.0 ** -53) + list(-odd * 2.0 ** -54))
