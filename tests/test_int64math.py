"""root_pair (csrc/int64math.cuh), the integer root and reciprocal root of the
Krylov scalars, in its host build against extended precision: about 2^-58
before one rounding to 53 bits each (2^-52.9); arguments that are not positive
normal numbers give what the FP64 functions give."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2209_15095_gb300", "csrc")
SRC = """
#include "int64math.cuh"
extern "C" void roots(int n, const double* a, double* s, double* r) {
  for (int i = 0; i < n; ++i) etd::root_pair(a[i], s[i], r[i]);
}
"""


@pytest.fixture(scope="module")
def roots(tmp_path_factory):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    d = tmp_path_factory.mktemp("int64math")
    (d / "r.cpp").write_text(SRC)
    subprocess.run([cxx, "-O2", "-shared", "-fPIC", "-I" + CSRC, str(d / "r.cpp"), "-o", str(d / "r.so")], check=True)
    lib = ctypes.CDLL(str(d / "r.so"))

    def call(a):
        a = np.ascontiguousarray(a, dtype=np.float64)
        s, r = np.empty_like(a), np.empty_like(a)
        lib.roots(a.size, *(x.ctypes.data_as(ctypes.c_void_p) for x in (a, s, r)))
        return s, r

    return call


def test_root_pair(roots):
    rng = np.random.default_rng(6)
    a = np.ldexp(1.0 + rng.random(20000), rng.integers(-1022, 1023, 20000))
    edge = [np.ldexp(1.0, k) for k in range(-1022, 1024)]
    edge += [np.nextafter(x, 0.0) for x in edge if x > 1e-300] + [np.finfo(np.float64).max]
    a = np.concatenate([a, edge])
    s, r = roots(a)
    ref = np.sqrt(a.astype(np.longdouble))
    assert np.max(np.abs(s / ref - 1)) <= 2.0 ** -52.9
    assert np.max(np.abs(r * ref - 1)) <= 2.0 ** -52.9


def test_root_pair_other_arguments(roots):
    a = np.array([0.0, -0.0, -1.0, np.inf, -np.inf, np.nan, 5e-324, 1e-310])
    s, r = roots(a)
    with np.errstate(invalid="ignore", divide="ignore"):
        ref = np.sqrt(a)
        np.testing.assert_array_equal(s, ref)
        np.testing.assert_array_equal(r, 1.0 / ref)
