"""The three-part single-precision sum of the gradient's hat rows, compiled for
the host, against exact rational sums: never further off than adding the same
128 numbers up in double may be."""
import ctypes
import os
import shutil
import subprocess
from fractions import Fraction

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SRC = r"""
#include "sums.h"
extern "C" double sum3(const float *x, int n)
{
    mcx::Sum3 t;
    for (int i = 0; i < n; ++i) t.add(x[i]);
    return t.value();
}
"""


@pytest.fixture(scope="module")
def sum3(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    d = tmp_path_factory.mktemp("sums")
    src, lib = d / "s.cpp", d / "s.so"
    src.write_text(SRC)
    subprocess.run([cxx, "-std=c++17", "-O2", "-shared", "-fPIC", "-Wall", "-Werror", "-I",
                    os.path.join(ROOT, "paper_2507_23189_gb300", "csrc"), "-o", str(lib), str(src)], check=True)
    f = ctypes.CDLL(str(lib)).sum3
    f.restype = ctypes.c_double
    return lambda x: f(x.ctypes.data_as(ctypes.POINTER(ctypes.c_float)), len(x))


@pytest.mark.parametrize("kind", ["uniform", "signed", "wide", "cancelling"])
def test_as_good_as_double(sum3, kind):
    rng = np.random.default_rng(7)
    worst = 0.0
    for _ in range(400):
        if kind == "uniform":
            x = rng.uniform(0, 1, 128)
        elif kind == "signed":
            x = rng.normal(size=128)
        elif kind == "wide":
            x = rng.normal(size=128) * 10.0 ** rng.uniform(-12, 12, 128)
        else:
            x = rng.normal(size=128) * 10.0 ** rng.uniform(0, 6, 128)
            x[64:] = -x[:64][::-1] * (1 + rng.uniform(-1e-6, 1e-6, 64))
        x = x.astype(np.float32)
        exact = sum((Fraction(float(v)) for v in x), Fraction(0))
        size = sum(abs(Fraction(float(v))) for v in x)
        worst = max(worst, float(abs(Fraction(sum3(x)) - exact) / size))
    # a running double sum: 127 additions that round to 2^-53
    assert worst <= 127 * 2.0 ** -53


def test_infinities_and_nan_pass(sum3):
    inf, nan = np.float32(np.inf), np.float32(np.nan)
    one = np.ones(5, np.float32)
    assert sum3(np.append(one, inf)) == np.inf and sum3(np.append(-inf, one)) == -np.inf
    assert np.isnan(sum3(np.append(one, nan))) and np.isnan(sum3(np.array([inf, -inf])))
