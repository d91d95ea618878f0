"""The range of the integer WENO5 form (csrc/weno_int.cuh): values up to 64h, as
the stencils of tube nodes reach where phi is not clamped (10h), and adjacent
differences in [-2^57, 2^57) units.

CPU: the host build.  Conversion is to nearest (half a unit); 12 Phi to the
bound of its own arithmetic (4 units and 2^-52 of the terms) up to the largest
differences.  GPU: steps of an unclamped phi on spacings with a large mantissa,
against the oracle at the step's 1e-10 h.
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
  for (int i = 0; i < n; ++i) out[i] = to_fix(f[i], k.eh, FIX_KMAX);
}
extern "C" void in_range(int n, const long long* F, int* out) {
  for (int i = 0; i < n; ++i) {
    i64 f[7], q[6];
    for (int k = 0; k < 7; ++k) f[k] = F[7 * i + k];
    out[i] = fix_diffs(f, q) < FIX_DIFF_HI && hi_mag(f[3]) < FIX_OWN_HI;
  }
}
extern "C" void phi12(int n, double h, const long long* e, long long* out) {
  const WenoInt k = weno_int(h, 1e-6);
  for (int i = 0; i < n; ++i) out[i] = weno_phi12(e[4 * i], e[4 * i + 1], e[4 * i + 2], e[4 * i + 3], k);
}
"""
OUT = 1 << 62


@pytest.fixture(scope="module")
def host(tmp_path_factory):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    d = tmp_path_factory.mktemp("wrange")
    (d / "w.cpp").write_text(SRC)
    subprocess.run([cxx, "-O2", "-shared", "-fPIC", "-I" + CSRC, str(d / "w.cpp"), "-o", str(d / "w.so")], check=True)
    return ctypes.CDLL(str(d / "w.so"))


def _p(a):
    return a.ctypes.data_as(ctypes.c_void_p)


@pytest.mark.parametrize("h", [1.0, 1.93, 12.0 / 199.0, 1.9999999, 3.7e5])
def test_conversion_and_range(host, h):
    rng = np.random.default_rng(5)
    n = 20000
    # a tube node's stencil of an unclamped distance: |phi| < 6h + one node's 4h
    f = np.ascontiguousarray(h * (6.0 * (2.0 * rng.random((n, 1)) - 1.0) + (2.0 * rng.random((n, 1)) - 1.0) * np.arange(-3, 4)))
    F = np.empty((n, 7), dtype=np.int64)
    host.fix(f.size, ctypes.c_double(h), _p(f), _p(F))
    U = np.ldexp(1.0, int(np.floor(np.log2(h))) - 54)
    assert np.all(np.abs(F.astype(np.longdouble) * U - f.astype(np.longdouble)) <= 0.5 * U)
    ok = np.empty(n, dtype=np.int32)
    host.in_range(n, _p(F), _p(ok))
    assert ok.all()
    # the ends: 128 2^eh, infinities, NaN, and small values to nearest
    top = np.ldexp(128.0, int(np.floor(np.log2(h))))
    f = np.array([top, -top, np.nextafter(top, 0.0), np.inf, -np.inf, np.nan, 0.4999 * U, 0.5 * U, U, -1.5 * U, 5e-324])
    F = np.empty(f.size, dtype=np.int64)
    host.fix(f.size, ctypes.c_double(h), _p(f), _p(F))
    assert list(F[:5]) == [OUT, -OUT, (1 << 61) - (1 << 8), OUT, -OUT] and abs(int(F[5])) == OUT
    assert list(F[6:]) == [0, 1, 1, -2, 0]


def test_out_of_range_values_are_seen(host):
    base = (1 << 61) - 1  # the largest value in range, next to every kind of neighbour
    rows, want = [], []  # differences are in range from -2^57 to 2^57 - 1
    for own in (0, base, -base):
        for v in (OUT, -OUT):
            for pos in (0, 1, 2, 4, 5, 6):
                r = [own] * 7
                r[pos] = v
                rows.append(r)
                want.append(0)
        m = 1 << 57
        for s, ok in ((m - 1, 1), (m, 0)) if own <= 0 else ((-m, 1), (-m - 1, 0)):
            rows.append([own, own, own, own, own + s, own + s, own + s])
            want.append(ok)
    for own in (OUT, -OUT):
        rows += [[own] * 7, [own] * 3 + [own] + [-own] * 3]
        want += [0, 0]
    F = np.array(rows, dtype=np.int64)
    got = np.empty(len(rows), dtype=np.int32)
    host.in_range(len(rows), _p(F), _p(got))
    assert got.tolist() == want


@pytest.mark.parametrize("h", [1.0, 1.9999999])
def test_phi12_at_the_largest_differences(host, h):
    rng = np.random.default_rng(8)
    m = (1 << 57) - 1
    sg = np.array([[(i >> k & 1) * 2 - 1 for k in range(6)] for i in range(64)], dtype=np.int64) * m
    q = np.concatenate([sg, rng.integers(-m, m, (20000, 6))])
    e = np.ascontiguousarray(np.diff(q, axis=1)[:, :4])
    got = np.empty(len(e), dtype=np.int64)
    host.phi12(len(e), ctypes.c_double(h), _p(e), _p(got))
    L = np.longdouble
    U = L(2.0) ** (int(np.floor(np.log2(h))) - 54)
    a, b, c, d = [e[:, i].astype(L) * U for i in range(4)]
    eps, k = L(4e-6) * L(h) ** 2, L(13) / 3
    s = [eps + k * (a - b) ** 2 + (a - 3 * b) ** 2, eps + k * (b - c) ** 2 + (b + c) ** 2,
         eps + k * (c - d) ** 2 + (3 * c - d) ** 2]
    A, B, C = [(s[i] * s[j]) ** 2 for i, j in ((1, 2), (0, 2), (0, 1))]
    X, Y = a - 2 * b + c, b - 2 * c + d
    ref = (4 * A * X + (3 * C - A - 6 * B) * Y) / (A + 6 * B + 3 * C)
    assert np.all(np.abs(got.astype(L) * U - ref) <= 4 * U + L(2.0) ** -52 * (4 * np.abs(X) + np.abs(Y)))


@pytest.mark.gpu
@pytest.mark.parametrize("precision,tol", [("fp64", 1e-10), ("mixed", 1e-2)])
@pytest.mark.parametrize("ndim,n", [(2, 34), (3, 34), (3, 67), (4, 18)])
def test_unclamped_step(ndim, n, precision, tol):
    """Two steps, the second with reinitialisation, of a distance that levelset_prepare
    has not clamped; h = 1.88 to 1.94 powers of 2, the tube's stencils reach 9h to 10h.
    The library clamps the nodes that it updates, the oracle every node: the others
    keep their values in between."""
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
    r = np.sqrt(sum((x[d] - 0.02 * d) ** 2 for d in range(ndim)))
    phi = r - 0.55 * box
    u = np.where(phi < 0, np.cos(r), 0.0)
    dt = 0.05 * g.h
    ctx = etd.Context(g.n, g.lo, g.hi, precision=precision)
    dphi = torch.tensor(phi, device="cuda")
    for reinit in (False, True):
        op = EBOperator(g, phi, 1.0)
        u = np.where(op.comp, u, 0.0)
        T = levelset.tube(phi, g.h)
        du = torch.tensor(u, device="cuda")
        ctx.init_domain(0, dphi)
        ctx.levelset_advance(0, dphi, du, dt, reinit)
        new, u, _ = levelset.levelset_advance(phi, u, op.comp, g, dt, 1.0, False)
        phi = np.where(T, new, phi)
    T = levelset.tube(phi, g.h)
    phi = np.where(T, levelset.clamp(levelset.reinit(phi, g.h), g.h), phi)
    ctx.sync()
    assert np.max(np.abs(dphi.cpu().numpy() - phi)) <= tol * g.h
