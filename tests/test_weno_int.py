"""The integer form of the HJ-WENO5 stages (csrc/weno_int.cuh).

CPU: its host build against extended precision.  With U = 2^-S <= 2^-54 h the
unit, 12 Phi is truncated a few times (4 units) and its weights are 64-bit
quantities truncated some ten times each (2^-52 of the terms they multiply);
the square root is rounded once to 53 bits after 2^-58 steps (2^-52.9).
GPU: level-set steps whose values leave the integer range (the kernel then
evaluates those nodes in FP64), on few and many nodes, against the oracle at
the step's 1e-10 h.
"""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2209_15095_gb300", "csrc")
SRC = """
#include <math.h>
#include "weno_int.cuh"
using namespace etd;
extern "C" void fix(int n, double h, const double* f, long long* out) {
  const WenoInt k = weno_int(h, 1e-6);
  for (int i = 0; i < n; ++i) out[i] = to_fix(f[i], k.eh);
}
extern "C" void phi12(int n, double h, const long long* e, long long* out) {
  const WenoInt k = weno_int(h, 1e-6);
  for (int i = 0; i < n; ++i) out[i] = weno_phi12(e[4 * i], e[4 * i + 1], e[4 * i + 2], e[4 * i + 3], k);
}
extern "C" void grad(int n, double h, const unsigned long long* a, double* out) {
  const WenoInt k = weno_int(h, 1e-6);
  for (int i = 0; i < n; ++i) out[i] = grad_of(U128{a[2 * i], a[2 * i + 1]}, k);
}
"""


@pytest.fixture(scope="module")
def host(tmp_path_factory):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    d = tmp_path_factory.mktemp("weno")
    (d / "w.cpp").write_text(SRC)
    subprocess.run([cxx, "-O2", "-shared", "-fPIC", "-I" + CSRC, str(d / "w.cpp"), "-o", str(d / "w.so")], check=True)
    return ctypes.CDLL(str(d / "w.so"))


def _p(a):
    return a.ctypes.data_as(ctypes.c_void_p)


def _stencils(rng, h, kind, n):
    """Seven consecutive values of phi per row."""
    x = np.arange(-3, 4) * h
    s = 2.0 * rng.random((n, 1)) - 1.0
    if kind == "rough":
        return h * (2.0 * rng.random((n, 7)) - 1.0) * 10.0 ** (-8.0 * rng.random((n, 1)))
    if kind == "smooth":
        return s * x + h * 10.0 ** (-6.0 * rng.random((n, 1))) * np.sin(0.3 * x / h + 6.0 * s)
    if kind == "clamped":
        return np.clip(s * x + 6.0 * h * (2.0 * rng.random((n, 1)) - 1.0), -6.0 * h, 6.0 * h)
    return np.abs(s * x + 0.5 * h * rng.random((n, 1))) - 0.3 * h  # kink


@pytest.mark.parametrize("kind", ["rough", "smooth", "clamped", "kink"])
@pytest.mark.parametrize("h", [1.0, 12.0 / 127.0, 1.9999999, 1e-4, 3.7e5])
def test_phi12_against_extended_precision(host, h, kind):
    n = 20000
    f = np.ascontiguousarray(_stencils(np.random.default_rng(3), h, kind, n))
    F = np.empty((n, 7), dtype=np.int64)
    host.fix(f.size, ctypes.c_double(h), _p(f), _p(F))
    U = np.ldexp(1.0, int(np.floor(np.log2(h))) - 54)
    assert np.all(np.abs(F.astype(np.longdouble) * U - f.astype(np.longdouble)) <= 0.5 * U)
    assert np.all(F.astype(np.float64) * U == f, where=np.abs(f) >= h / 4)
    e = np.ascontiguousarray(np.diff(np.diff(F, axis=1), axis=1)[:, :4])
    got = np.empty(n, dtype=np.int64)
    host.phi12(n, ctypes.c_double(h), _p(e), _p(got))
    a, b, c, d = [e[:, i].astype(np.longdouble) * U for i in range(4)]
    eps = np.longdouble(4e-6) * np.longdouble(h) ** 2
    k = np.longdouble(13) / 3
    s = [eps + k * (a - b) ** 2 + (a - 3 * b) ** 2, eps + k * (b - c) ** 2 + (b + c) ** 2,
         eps + k * (c - d) ** 2 + (3 * c - d) ** 2]
    A, B, C = [(s[i] * s[j]) ** 2 for i, j in ((1, 2), (0, 2), (0, 1))]
    X, Y = a - 2 * b + c, b - 2 * c + d
    ref = (4 * A * X + (3 * C - A - 6 * B) * Y) / (A + 6 * B + 3 * C)
    bound = 4 * U + 2.0 ** -52 * (4 * np.abs(X) + np.abs(Y))
    assert np.all(np.abs(got.astype(np.longdouble) * U - ref) <= bound)


def test_fix_out_of_range(host):
    h = 0.3  # 2^-2 <= h: the range ends at 16 2^-2 = 4
    f = np.array([4.0, -4.0, np.nextafter(4.0, 0.0), np.inf, -np.inf, np.nan, 1e300, 0.0, -0.0, 5e-324])
    F = np.empty(f.size, dtype=np.int64)
    host.fix(f.size, ctypes.c_double(h), _p(f), _p(F))
    out = 1 << 62
    assert list(F[:2]) == [out, -out] and abs(F[2]) < 1 << 58
    assert F[3] == out and F[4] == -out and abs(F[5]) == out and F[6] == out and not F[7:].any()
    one = np.ones(1)
    host.fix(1, ctypes.c_double(1e-290), _p(one), _p(F))
    assert F[0] == out


def test_gradient_root(host):
    rng = np.random.default_rng(4)
    v = [0, 1, 2, 3, (1 << 64) - 1, 1 << 64, 1 << 125, 1 << 126, (1 << 127) - 1]
    v += [int(rng.integers(1 << 62)) * (1 << int(s)) + int(rng.integers(1 << 30)) for s in rng.integers(0, 64, 2000)]
    v += [int(rng.integers(1 << 62)) >> int(s) for s in rng.integers(0, 62, 500)]
    a = np.array([[x >> 64, x & ((1 << 64) - 1)] for x in map(int, v)], dtype=np.uint64)
    got = np.empty(len(v))
    h = 0.7
    host.grad(len(v), ctypes.c_double(h), _p(a), _p(got))
    ref = np.sqrt(np.array([np.longdouble(x >> 64) * np.longdouble(2) ** 64 + np.longdouble(x & ((1 << 64) - 1))
                            for x in map(int, v)])) * np.longdouble(2.0 ** -55) / (12 * np.longdouble(h))
    # the root to 2^-52.9, the scale's two roundings and the product's one
    assert np.all(np.abs(got - ref) <= 2.0 ** -51 * ref)


@pytest.mark.gpu
@pytest.mark.parametrize("ndim,n", [(2, 40), (3, 24), (3, 97), (4, 16)])
@pytest.mark.parametrize("slope", [1.0, 3.0, 9.0])
def test_step_out_of_integer_range(ndim, n, slope):
    """Advection of phi = slope (r - R), not clamped: at slope 3 the nodes
    beyond the band leave the range, at slope 9 nodes of the band do; on few
    nodes (an axis per lane) and many (a node per lane: 3D at 97)."""
    import torch

    from oracle import levelset
    from oracle.eb import EBOperator
    from oracle.grid import Grid
    from paper_2209_15095_gb300 import build

    build.build()
    from paper_2209_15095_gb300 import etd

    box = 2.0
    g = Grid((n,) * ndim, (-box,) * ndim, (box,) * ndim)
    x = g.coords()
    r = np.sqrt(sum(((x[d] - 0.02 * d) / (1.0 + 0.05 * d)) ** 2 for d in range(ndim)))
    phi = slope * (r - 0.55 * box)
    u = np.where(phi < 0, np.cos(r), 0.0)
    dt = 0.05 * g.h
    op = EBOperator(g, phi, 1.0)
    u = np.where(op.comp, u, 0.0)
    ref_phi, ref_u, _ = levelset.levelset_advance(phi, u, op.comp, g, dt, 1.0, False)
    ctx = etd.Context(g.n, g.lo, g.hi, precision="fp64")
    dphi = torch.tensor(phi, device="cuda")
    du = torch.tensor(u, device="cuda")
    ctx.init_domain(0, dphi)
    ctx.levelset_advance(0, dphi, du, dt, False)
    ctx.sync()
    T = levelset.tube(phi, g.h)  # the nodes that the step updates
    assert np.max(np.abs(dphi.cpu().numpy() - ref_phi)[T]) <= 1e-10 * g.h
