"""The sum that ends the Jacobi steps of PageRank, |pr' - pr| over the rows that
the threads finish, compiled for the host: no further from the exact sum than
one kept in 64 bits."""
import ctypes
import os
import subprocess
from fractions import Fraction

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2507_11094_gb300", "csrc")
SRC = r"""
#include "sp_acc.cuh"
extern "C" double run(const float *a, const float *b, int n) {
  sp::Acc c, d;   // two threads' shares, merged
  for (int i = 0; i < n; ++i) sp::acc_diff(i % 2 ? d : c, a[i], b[i]);
  sp::acc_merge(c, d);
  return sp::acc_value(c);
}
"""


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    d = tmp_path_factory.mktemp("acc")
    (d / "acc.cpp").write_text(SRC)
    lib = d / "acc.so"
    subprocess.run(["g++", "-std=c++17", "-O2", "-shared", "-fPIC", "-I", CSRC,
                    str(d / "acc.cpp"), "-o", str(lib)], check=True)
    f = ctypes.CDLL(str(lib)).run
    f.restype = ctypes.c_double
    fp = np.ctypeslib.ndpointer(np.float32, flags="C_CONTIGUOUS")
    f.argtypes = [fp, fp, ctypes.c_int]
    return f


def exact(a, b):
    return sum((abs(Fraction(float(x)) - Fraction(float(y))) for x, y in zip(a, b)), Fraction(0))


# values as far apart as a rank and its neighbours' ranks are, alike or not,
# zeros, and more rows than a thread ever finishes of 2^31 vertices.  The value
# is a double, so half a unit of its last place (2^-53) is lost at the end; what
# the float sums lose before is below 4 k^3 2^-72 of the sum for k rows in the
# worst case and far less for the mixed signs of real errors: under 2^-55 here.
@pytest.mark.parametrize("k", [1, 2, 7, 64, 1000])
@pytest.mark.parametrize("kind", ["ranks", "far", "alike", "zeros", "falling"])
def test_sum_of_differences(run, k, kind):
    rng = np.random.default_rng(k)
    for _ in range(20):
        a = rng.random(k) / 1e6
        b = rng.random(k) / 1e6
        if kind == "far":
            a = a * 10.0 ** rng.integers(-12, 6, k)
        elif kind == "alike":
            b = a * (1 + rng.normal(size=k) * 1e-6)
        elif kind == "zeros":
            a[rng.random(k) < 0.5] = 0
            b[rng.random(k) < 0.5] = 0
        elif kind == "falling":
            a = 0.5 ** (2.0 * np.arange(k) % 60)
            b = a * rng.random(k)
        a, b = np.ascontiguousarray(a, np.float32), np.ascontiguousarray(b, np.float32)
        want = exact(a, b)
        got = Fraction(run(a, b, k))
        assert abs(got - want) <= want * (Fraction(1, 2 ** 53) + Fraction(1, 2 ** 55))
        plain = np.float64(0)
        for x, y in zip(a, b):
            plain += abs(np.float64(x) - np.float64(y))
        assert abs(got - want) <= abs(Fraction(float(plain)) - want) + want / 2 ** 53
