"""The Chebyshev table of the small exponential (csrc/cheb.cuh), part of the module.

CPU: the compiler's table against 40-digit values.  Each step of the recurrence
rounds three times and adds positive terms, so a value is off by 3 roundings for
every step above it at most, the normalising sum by as much and its own 512: 2050
roundings of 2^-53.
No table is filled by a copy on first use, which would serve one device and one
stream's order only.  GPU: the first Krylov launch of a process, under stream
capture, gives what a plain one gives.
"""
import ctypes
import os
import shutil
import subprocess
import sys

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2209_15095_gb300", "csrc")
SRC = """
#include "cheb.cuh"
constexpr etd::ChebTables T = etd::cheb_tables();
static_assert(T.at[etd::CHEB_TABLES] == etd::CHEB_MAX, "the table fits");
extern "C" int get(double* c, double* two_a, int* at) {
  for (int i = 0; i < etd::CHEB_MAX; ++i) c[i] = T.c[i];
  for (int i = 0; i < etd::CHEB_TABLES; ++i) two_a[i] = T.two_a[i];
  for (int i = 0; i <= etd::CHEB_TABLES; ++i) at[i] = T.at[i];
  return etd::CHEB_TABLES;
}
"""
CAPTURED = """
import sys
sys.path.insert(0, sys.argv[1])
import torch
from paper_2209_15095_gb300 import etd
n = 40
x = torch.linspace(-1.0, 1.0, n, dtype=torch.float64, device="cuda")
r = (x[:, None] ** 2 + x[None, :] ** 2).sqrt()
phi = (r - 0.6).contiguous()
v = [torch.cos((k + 1.0) * r).contiguous() for k in range(3)]
y, z = torch.zeros_like(phi), torch.zeros_like(phi)
s = torch.cuda.Stream()
s.wait_stream(torch.cuda.current_stream())
with torch.cuda.stream(s):
    ctx = etd.Context((n, n), (-1.0, -1.0), (1.0, 1.0))
    ctx.init_domain(0, phi)
torch.cuda.synchronize()
g = torch.cuda.CUDAGraph()
with torch.cuda.graph(g, stream=s):
    ctx.phi_combination(0, 0.01, *v, y)
g.replay()
torch.cuda.synchronize()
with torch.cuda.stream(s):
    ctx.phi_combination(0, 0.01, *v, z)
ctx.sync()
assert z.abs().max() > 0.1 and torch.equal(y, z)
print("same")
"""


def test_table(tmp_path):
    mp = pytest.importorskip("mpmath")
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    (tmp_path / "c.cpp").write_text(SRC)
    subprocess.run([cxx, "-std=c++17", "-O2", "-shared", "-fPIC", "-I" + CSRC, str(tmp_path / "c.cpp"), "-o",
                    str(tmp_path / "c.so")], check=True)
    c, two_a, at = np.empty(4096), np.empty(64), np.empty(64, dtype=np.int32)
    n = ctypes.CDLL(str(tmp_path / "c.so")).get(*(x.ctypes.data_as(ctypes.c_void_p) for x in (c, two_a, at)))
    mp.mp.dps = 40
    for i in range(n):
        a = mp.mpf(2) ** (mp.mpf(i) / 2)
        assert abs(mp.mpf(two_a[i]) * a / 2 - 1) < 2.0 ** -51
        m = at[i + 1] - at[i]
        ref = [2 * mp.exp(-a) * mp.besseli(k, a) for k in range(m + 1)]
        assert ref[m] < 1.0001e-24
        for k in range(m):
            assert abs(mp.mpf(c[at[i] + k]) / ref[k] - 1) <= 2050 * 2.0 ** -53


def test_no_table_is_filled_by_a_copy():
    for f in os.listdir(CSRC):
        with open(os.path.join(CSRC, f)) as h:
            assert "cudaMemcpyToSymbol" not in h.read(), f


@pytest.mark.gpu
def test_first_launch_under_capture():
    from paper_2209_15095_gb300 import build

    build.build()
    r = subprocess.run([sys.executable, "-c", CAPTURED, ROOT], capture_output=True, text=True)
    assert r.returncode == 0 and r.stdout.strip() == "same", r.stderr[-2000:]
